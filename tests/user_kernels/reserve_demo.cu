// A user kernel that reserves queue slots with a reservation word read earlier: one thread
// reads the word, another command takes the slot it names, then the thread reserves with
// the old word.  Only a queue that is full may refuse it.
#include <cstdint>

#include "agile_device.cuh"

namespace {

struct ReserveDemo {
  uint32_t n;
  int32_t *got;  // per round: the reservation with the old word succeeded

  // reserve a slot of queue 0 and spend it on a no-op command
  __device__ static bool no_op(const agile::Dev &d, uint64_t word) {
    uint32_t q = 0, slot = 0, ticket = 0;
    if (!agile::sq_reserve_dev(d, 0, 0, 1, q, slot, ticket, false, word)) return false;
    agile::sq_write(d, q, slot, ticket, agile::OP_FLUSH, 0, 0, agile::ctx_make(agile::CTX_NOP, 0, 0));
    agile::sq_ring(d, q, ticket);
    return true;
  }

  __device__ void run(const agile::Dev &d, const agile::AppCtx &a) const {
    if (a.warp != 0 || (threadIdx.x & 31) != 0) return;
    for (uint32_t i = 0; i < n; ++i) {
      // the earlier commands have completed (waited for with a bound)
      const uint64_t end = agile::dev::now() + 100'000'000;
      while ((agile::ld_rlx64(&d.sq_resv[0]) >> 32) != 0 && agile::dev::now() < end) __nanosleep(200);
      const uint64_t old_word = agile::sq_first_word(d, 0, 0, false);
      got[i] = no_op(d, agile::kNoWord) && no_op(d, old_word) ? 1 : 0;
    }
  }
};

}  // namespace

extern "C" int reserve_demo(agile_ctx *ctx, uint32_t n, int32_t *got, void *stream) {
  ReserveDemo app{n, got};
  return agile::launch_user(ctx, app, stream, 1);
}
