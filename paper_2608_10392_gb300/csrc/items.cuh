// The order in which CTAs take the work items of a tiled kernel.
#pragma once

namespace unif {

// Items (tile, part), `parts` of them per tile, dealt out in turn to `ctas`
// CTAs: CTA `cta` takes items cta, cta + ctas, ... counted tile by tile. Their
// number may be beyond 32 bits, each coordinate is not.
struct ItemWalk {
  int tile, part;

  __host__ __device__ __forceinline__ ItemWalk(int cta, int ctas, int parts)
      : tile(cta / parts), part(cta % parts), parts_(parts), tiles_on_(ctas / parts),
        parts_on_(ctas % parts) {}
  __host__ __device__ __forceinline__ void next() {
    tile += tiles_on_;
    part += parts_on_;
    if (part >= parts_) {
      part -= parts_;
      ++tile;
    }
  }

 private:
  int parts_, tiles_on_, parts_on_;
};

}  // namespace unif
