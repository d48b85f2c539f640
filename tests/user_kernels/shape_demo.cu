// A user kernel that keeps something for each warp of its CTA in shared memory, sized by
// agile::kWarps: every warp checks its index, leaves a mark in its place and reads it back
// after the CTA's other warps have left theirs.
#include <cstdint>

#include "agile_device.cuh"

namespace {

struct ShapeDemo {
  uint32_t *outside;  // warps whose index or CTA does not fit
  uint32_t *lost;     // marks overwritten
  uint32_t *seen;     // [n_warps] + 1 per warp index

  __device__ void run(const agile::Dev &d, const agile::AppCtx &a) const {
    __shared__ uint32_t mark[agile::kWarps][32];
    const uint32_t w = threadIdx.x / 32, l = threadIdx.x & 31;
    if (w >= agile::kWarps || blockDim.x != agile::kThreads) {
      if (l == 0) atomicAdd(outside, 1u);
      return;
    }
    mark[w][l] = a.warp * 32 + l;
    if (!agile::dev::barrier(d, a)) return;
    if (*(volatile uint32_t *)&mark[w][l] != a.warp * 32 + l) atomicAdd(lost, 1u);
    if (l == 0) atomicAdd(&seen[a.warp], 1u);
  }
};

}  // namespace

extern "C" int shape_demo(agile_ctx *ctx, uint32_t *outside, uint32_t *lost, uint32_t *seen, uint32_t app_warps,
                          void *stream) {
  ShapeDemo app{outside, lost, seen};
  return agile::launch_user(ctx, app, stream, app_warps);
}
