// Device-side state and primitives of the AGILE I/O path for sm_103a.
//
// Layout in HBM (all library-owned, allocated once per context):
//   lines      [nlines * 4096]      cache data, one 4 KiB line per store page (Sec. 2.3.3)
//   tag        [nlines] u64         {page:44 | pin:16 | wb:1 | ref:1 | state:2} (Sec. 3.4)
//   hand       [sets]   u32         clock hand per set (Sec. 4.4, clock policy)
//   sh_key     [buckets] u64        in-flight share table, 4 slots of 16 bits per bucket
//   sh_val     [buckets*4] u64      (Sec. 3.4.1), and the token of each slot's read
//   sq         [Q * depth] 64 B     NVMe submission entries (Sec. 2.1)
//   cq         [Q * 2*depth] 16 B   NVMe completion entries with phase bit (Sec. 2.1)
//   sqe_state  [Q * depth] u64      {ticket:62 | EMPTY/UPDATED/WRITTEN} (Sec. 3.3.1)
//   cmd_ctx    [Q * depth] u64      what a completion releases (line fill, write-back)
//   cmpl       [Q * depth] u64      completion word = transaction barrier (Sec. 3.2.1)
//   sq_resv    [Q] u64              {in flight:32 | next ticket:32}
//   sq_db      [Q] u32              doorbell: commands issued so far (slot = count mod depth)
//   cq_db      [Q] u32              CQ head doorbell
//   cq_poll    [Q*4] u32            Alg. 1 state {offset, mask, phase}
//   emu_*      [Q] u32              emulated device: fetch/seen/CQ-slot counters, timing
//   staging    [Q * depth * 4096]   write-back sources, one page per submission slot
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace agile {

constexpr uint32_t kPage = 4096;
// A CTA of a user kernel (agile::launch_user) has kWarps warps, as many CTAs on an SM as its
// application is compiled for (MinBlocks, 2 by default: 16 warps of 128 registers an SM).
// A library call's engine has the same warps in one CTA.
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- tag word (Sec. 3.4)
constexpr uint64_t ST_MASK = 3, ST_INVALID = 0, ST_BUSY = 1, ST_READY = 2, ST_MODIFIED = 3;
constexpr uint64_t TAG_REF = 1ull << 2;
constexpr uint64_t TAG_WB = 1ull << 3;
constexpr int PIN_SHIFT = 4;
constexpr uint64_t PIN1 = 1ull << PIN_SHIFT;
constexpr uint64_t PIN_MASK = 0xFFFFull << PIN_SHIFT;
constexpr int PAGE_SHIFT = 20;
__host__ __device__ __forceinline__ uint64_t tag_page(uint64_t t) { return t >> PAGE_SHIFT; }
__host__ __device__ __forceinline__ uint64_t tag_state(uint64_t t) { return t & ST_MASK; }
__host__ __device__ __forceinline__ uint64_t tag_make(uint64_t page, uint64_t st, bool ref) {
  return (page << PAGE_SHIFT) | (ref ? TAG_REF : 0) | st;
}

// replacement policies (agile.h AGILE_POLICY_*)
constexpr uint32_t kPolicyClock = 0, kPolicyFifo = 1;

// ---------------------------------------------------------------- queues (Sec. 3.3.1)
constexpr uint64_t SQE_EMPTY = 0, SQE_UPDATED = 1, SQE_WRITTEN = 2;
constexpr uint32_t OP_FLUSH = 0x00, OP_WRITE = 0x01, OP_READ = 0x02;

// command context: what the completion of a command releases (CTX_BUF: a read into a
// user buffer, which releases only the page's in-flight entry)
constexpr uint64_t CTX_NOP = 0, CTX_FILL = 1, CTX_WB = 2, CTX_BUF = 3;
__host__ __device__ __forceinline__ uint64_t ctx_make(uint64_t kind, uint32_t share_slot, uint32_t idx) {
  return (kind << 60) | ((uint64_t)(share_slot & 0x0FFFFFFFu) << 32) | idx;
}

struct alignas(64) Sqe { uint32_t dw[16]; };
struct alignas(16) Cqe { uint32_t dw[4]; };

// statistic slots (mirror agile_stats_t order)
enum Stat {
  S_HITS, S_MISSES, S_BUSY_HITS, S_WARP_COALESCED, S_SHARE_RETRIES, S_EVICTIONS, S_WRITEBACKS,
  S_EAGAIN, S_SQ_FULL, S_DOORBELLS, S_COMMANDS, S_CQES, S_CQ_DOORBELLS, S_IO_ERRORS,
  S_BYTES_READ, S_BYTES_WRITTEN, S_PREFETCHES, S_TIMEOUTS, S_COUNT
};

// per-launch state, zeroed before every launch (and numbered) by run_reset_kernel
struct RunState {
  uint32_t app_done;      // CTAs whose application warps have all finished
  uint32_t error;         // first error code (negated AGILE_E*), 0 = none
  uint32_t bar_count;     // grid barrier arrivals (CTAs)
  uint32_t bar_gen;       // grid barrier generation
  uint32_t work[4];       // dynamic work counters
  unsigned long long acc[4];  // accumulators (edges scanned, discovered vertices, ...)
  uint32_t flag[4];
  uint32_t pending;       // bags the resident pass of a lookup has left to the engine
  uint32_t pad;
  unsigned long long epoch;  // number of this launch among the device's launches (never 0)
  // BFS slice queue, per level parity, each on a line of its own (hot words)
  alignas(128) uint32_t hub_count[2];  // slices of long adjacency lists reserved
  alignas(128) uint32_t hub_cursor[2];  // next slice ticket
  alignas(128) uint32_t units_done[2];  // CTAs whose warps have all finished their own vertices
};

// One command as the emulated device served it (times from %globaltimer, ns).
struct TraceRec {
  unsigned long long page;    // store page of the command
  unsigned long long t_seen;  // doorbell that exposed it first read by the device (0 when
                              // the device runs without a latency or throughput model)
  unsigned long long t_start; // taken by an engine: data movement starts
  unsigned long long t_done;  // completion entry posted
  uint32_t q, cid, opcode, status;
  unsigned long long t_commit;  // the command was written to its submission slot
  uint32_t pad[2];
};

struct Dev {
  // backing store (pinned host memory, device-visible address)
  uint8_t *store;
  uint64_t store_bytes;
  // cache
  uint8_t *lines;
  unsigned long long *tag;
  uint32_t *hand;
  uint64_t nlines;
  uint32_t sets, ways;
  unsigned long long *sh_key;
  unsigned long long *sh_val;
  uint32_t sh_bits;  // log2 of buckets * 2^15: the page numbers the table tells apart
  uint64_t sh_mul;   // odd: page * sh_mul mod 2^sh_bits = {bucket, 15-bit key}
  // queues
  uint32_t Q, depth, dmask, dlog;
  uint32_t Qp;       // queues [Q - Qp, Q) carry prefetches, served after the demand queues
  uint32_t cq_size;  // CQ entries per queue = 2 * depth
  Sqe *sq;
  Cqe *cq;
  unsigned long long *sqe_state;
  unsigned long long *cmd_ctx;
  unsigned long long *cmpl;
  unsigned long long *sq_resv;
  uint32_t *sq_db, *cq_db, *cq_poll;
  // device counters per queue, unwrapped: next command to fetch, doorbell seen, next CQ
  // slot (arrays of their own: engines scan the first one next to the doorbells)
  uint32_t *emu_fetch, *emu_seen, *emu_cqt;
  unsigned long long *emu_busy;     // [Q] ns at which the queue's device pipe is free
  unsigned long long *emu_arrival;  // [Q*depth] ns at which the device saw the command
  uint8_t *staging;
  // per store page: reads and writes the device served, dirty epochs the cache opened
  // (a clean line turned MODIFIED, or a write-through issued); every dirty epoch ends in
  // exactly one write
  uint32_t *pg_reads, *pg_writes, *pg_dirty;
  // command trace (optional): one record per command the device served
  struct TraceRec *trace;
  uint32_t trace_cap;
  uint32_t *trace_n;
  // application event log (optional, same capacity): {time, warp | kind << 32 | arg << 40}
  unsigned long long *ev;
  uint32_t *ev_n;
  // Share Table of user buffers (Sec. 3.4.1): 4 slots per bucket; key = page + 1,
  // buf = the buffer's address, meta = {state:8 | count:32 | closing:1}, tok = the token
  // of the read that fills the buffer (valid once the entry has left PENDING)
  unsigned long long *ub_key, *ub_buf, *ub_meta, *ub_tok;
  uint32_t ub_mask;  // buckets - 1; ub_key == nullptr: no Share Table
  // backing devices: page p lives on device p mod ndev at block p / ndev; queue q
  // belongs to device q mod ndev (Sec. 4.3: requests interleaved over the SSDs)
  uint32_t ndev;
  // replacement policy of the cache (AGILE_POLICY_*)
  uint32_t policy;
  // emulated device model
  uint64_t lat_ns, ns_per_page;
  uint64_t ns_rd_dev, ns_wr_dev;    // per-device time of one page read / written (0 = no cap)
  unsigned long long *dev_busy;     // [ndev] ns up to which the device is booked
  uint32_t fault_flags, fault_thresh;
  uint64_t seed;
  // run
  RunState *run;
  unsigned long long *stats;
  uint64_t timeout_ns;
  uint32_t prefetch_depth;
  int32_t *err_sticky;  // first error since the last agile_check
  uint32_t app_active;  // application warps that take part in this launch (0 = all)
  uint32_t extra_engines;  // idle application warps that may also serve the device
  uint64_t session_ns;  // length of a long-running launch (serving loop); 0 = timeout_ns
};

// What an engine CTA keeps in shared memory.
// dev: the launch's Dev, for the functions that are kept out of line.  They cannot read
// the kernel's parameter bank, and through a pointer to it every field would be a load
// that each fence sends back to L2 (issuing a command took 5.5 us that way, most of it
// such reloads).
struct CtaState {
  Dev dev;
  uint32_t done;                     // application warps of this CTA that have finished
  uint32_t bar_count, bar_gen;       // grid barrier: arrivals in this CTA, generation
  uint32_t active;                   // application warps of this CTA that take part
  uint32_t ctas_active;              // CTAs with such warps
  // slice queue (BFS, SpMV): warps of this CTA done with their own rows, and what the
  // CTA's watching warp has seen of the queue (end_seen: phase + 1 once every warp of the
  // grid is done and `end_count` slices are all there will be)
  uint32_t own_done, watched, end_seen, end_count;
};
__device__ __forceinline__ CtaState &cta_state() {
  __shared__ CtaState cs;
  return cs;
}
__device__ __forceinline__ const Dev &shared_dev() { return cta_state().dev; }

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t ld_acq32(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_acq64(const unsigned long long *p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_rlx32(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_rlx64(const unsigned long long *p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_rel32(uint32_t *p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_rel64(unsigned long long *p, uint64_t v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_rlx64(unsigned long long *p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_rlx32(uint32_t *p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t atom_add_acq(unsigned long long *p, uint64_t v) {
  uint64_t old;
  asm volatile("atom.acquire.gpu.global.add.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
  return old;
}
__device__ __forceinline__ uint64_t atom_cas_acq(unsigned long long *p, uint64_t cmp, uint64_t v) {
  uint64_t old;
  asm volatile("atom.acquire.gpu.global.cas.b64 %0, [%1], %2, %3;" : "=l"(old) : "l"(p), "l"(cmp), "l"(v) : "memory");
  return old;
}
__device__ __forceinline__ void fence_sc() { asm volatile("fence.sc.gpu;" ::: "memory"); }
__device__ __forceinline__ void fence_ar() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// 16-byte loads/stores that bypass L1: cache lines and store pages are rewritten by
// other SMs during a launch, so nothing here may be served from a stale L1 copy.
__device__ __forceinline__ int4 ld_cg16(const void *p) {
  int4 v;
  asm volatile("ld.global.cg.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_cg16(void *p, int4 v) {
  asm volatile("st.global.cg.v4.s32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w) : "memory");
}
__device__ __forceinline__ float4 ld_cg_f4(const void *p) {
  int4 v = ld_cg16(p);
  return make_float4(__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z), __int_as_float(v.w));
}
__device__ __forceinline__ int32_t ld_cg_s32(const void *p) {
  int32_t v;
  asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int64_t ld_cg_s64(const void *p) {
  int64_t v;
  asm volatile("ld.global.cg.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31; }

// counters are kept in kStatShards copies (by CTA) so that warps all over the GPU do not
// serialise on one address; the host adds the copies up
constexpr int kStatShards = 32;
__device__ __forceinline__ unsigned long long *stat_ptr(const Dev &d, int s) {
  return &d.stats[(blockIdx.x % kStatShards) * S_COUNT + s];
}

__device__ __forceinline__ void stat_add(const Dev &d, int s, uint64_t v) {
  if (v) atomicAdd(stat_ptr(d, s), (unsigned long long)v);
}
// warp-aggregated statistic: every lane passes its own count
__device__ __forceinline__ void stat_warp(const Dev &d, int s, uint32_t v) {
  unsigned b = __ballot_sync(kFull, v != 0);
  if (!b) return;
  uint32_t sum = __reduce_add_sync(kFull, v);
  if (lane_id() == 0) atomicAdd(stat_ptr(d, s), (unsigned long long)sum);
}

// Application event (lane 0 of a warp; only with the trace on): `kind` names the
// event, `arg` a small number (a level, ...).
__device__ __forceinline__ void app_event(const Dev &d, uint32_t warp, uint32_t kind, uint32_t arg) {
  if (!d.ev) return;
  uint32_t i = atomicAdd(d.ev_n, 1u);
  if (i < d.trace_cap) {
    d.ev[2 * i] = gtimer();
    d.ev[2 * i + 1] = (uint64_t)warp | ((uint64_t)(kind & 0xFF) << 32) | ((uint64_t)(arg & 0xFFFFFF) << 40);
  }
}

// A cache line of `page` turned from clean to MODIFIED (or a write-through was issued):
// the page owes the store one write.
__device__ __forceinline__ void note_dirty(const Dev &d, uint64_t page) {
  atomicAdd(&d.pg_dirty[page], 1u);
}

// record the first error of the launch and of the context
__device__ __forceinline__ void set_error(const Dev &d, int code) {
  atomicCAS(&d.run->error, 0u, (uint32_t)(-code));
  atomicCAS((uint32_t *)d.err_sticky, 0u, (uint32_t)(-code));
  if (code == -110) atomicAdd(stat_ptr(d, S_TIMEOUTS), 1ull);
}
__device__ __forceinline__ bool aborted(const Dev &d) { return ld_rlx32(&d.run->error) != 0; }

__device__ __forceinline__ void backoff(uint32_t &ns, uint32_t cap = 2048) {
  __nanosleep(ns);
  ns = ns < cap ? ns * 2 : cap;
}

// ---------------------------------------------------------------- cache geometry
// Set index: golden-ratio multiplicative hash of the page, upper 32 bits scaled to
// [0, sets).  Works for any number of sets.
__host__ __device__ __forceinline__ uint32_t set_of(uint64_t page, uint32_t sets) {
  uint64_t h = page * 0x9E3779B97F4A7C15ull;
  return (uint32_t)(((h >> 32) * (uint64_t)sets) >> 32);
}
__device__ __forceinline__ uint8_t *line_ptr(const Dev &d, uint64_t line) {
  return d.lines + line * (uint64_t)kPage;
}

// ---------------------------------------------------------------- warp page copy
// One warp moves one 4 KiB page with 16-byte accesses: 8 loads in flight per lane,
// then 8 stores, so each request is a single 512-byte coalesced transaction per step.
__device__ __forceinline__ void warp_copy_page(void *dst, const void *src) {
  const int4 *s = (const int4 *)src;
  int4 *t = (int4 *)dst;
  unsigned l = lane_id();
  int4 v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = ld_cg16(s + k * 32 + l);
#pragma unroll
  for (int k = 0; k < 8; ++k) st_cg16(t + k * 32 + l, v[k]);
}
// A single thread moves a page (rare paths: write-back copies inside a lane's miss).
__device__ __forceinline__ void lane_copy_page(void *dst, const void *src) {
  const int4 *s = (const int4 *)src;
  int4 *t = (int4 *)dst;
  for (int k = 0; k < 256; k += 16) {
    int4 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = ld_cg16(s + k + j);
#pragma unroll
    for (int j = 0; j < 16; ++j) st_cg16(t + k + j, v[j]);
  }
}

// ================================================================ submission side
// Alg. 2, check_full: reserve n consecutive slots of queue q.  A slot is free when
// the command that used it last has completed (state EMPTY) and fewer than depth-1
// commands are outstanding (the NVMe full rule).  Never waits.
// `w`: the queue's reservation word; `old_word`: it was read a while ago, and another command may
// have taken the slot it names since, so it is read again before the queue is taken for full.
// (A word just read is believed: reading it again while completions change it cost a flush
// of 85 k lines through full queues 7%.)
__device__ __forceinline__ bool sq_try_reserve(const Dev &d, uint32_t q, uint32_t n, uint64_t w, bool old_word,
                                               uint32_t &slot, uint32_t &ticket) {
  unsigned long long *rp = &d.sq_resv[q];
  for (int tries = 0; tries < 4; ++tries) {
    uint32_t t = (uint32_t)w, infl = (uint32_t)(w >> 32);
    bool room = infl + n <= d.depth - 1;
    for (uint32_t k = 0; k < n && room; ++k) {
      uint64_t st = ld_acq64(&d.sqe_state[(uint64_t)q * d.depth + ((t + k) & d.dmask)]);
      room = (st & 3) == SQE_EMPTY;
    }
    if (!room) {
      if (!old_word) return false;
      old_word = false;
      w = ld_rlx64(rp);
      continue;
    }
    old_word = false;
    uint64_t nw = ((uint64_t)(infl + n) << 32) | (uint32_t)(t + n);
    uint64_t old = atomicCAS(rp, (unsigned long long)w, (unsigned long long)nw);
    if (old == w) {
      slot = t & d.dmask;
      ticket = t;
      return true;
    }
    w = old;
  }
  return false;
}

// Backing device of a store page and its block number there (4 KiB blocks).
__host__ __device__ __forceinline__ uint32_t dev_of_page(const Dev &d, uint64_t page) {
  return d.ndev > 1 ? (uint32_t)(page % d.ndev) : 0u;
}
__host__ __device__ __forceinline__ uint64_t block_of_page(const Dev &d, uint64_t page) {
  return d.ndev > 1 ? page / d.ndev : page;
}

// SQ selection (Sec. 3.3.1): among the queues of the page's device in the request's
// class -- demand queues [0, Q - Qp), prefetch queues [Q - Qp, Q) (NVMe-style
// arbitration: the device serves demand queues first, so requests made ahead of need
// only use device time that demand leaves idle) -- start at the one nearest the
// thread's own queue, on a full queue try the class's next one of the device; false
// after one pass over them.
struct SqPick {
  uint32_t base, per, nd, k0;  // queue of the class's k-th of the device: base + k * nd + dv
};
__device__ __forceinline__ SqPick sq_pick(const Dev &d, uint32_t q0, bool pf) {
  SqPick p;
  p.nd = d.ndev > 1 ? d.ndev : 1u;
  p.base = pf && d.Qp ? d.Q - d.Qp : 0u;
  const uint32_t cnt = d.Qp ? (pf ? d.Qp : d.Q - d.Qp) : d.Q;
  if (p.nd == 1) {
    p.per = cnt;
    p.k0 = q0 < cnt ? q0 : q0 % cnt;
  } else {
    p.per = cnt / p.nd;  // queues of one device in the class
    p.k0 = (q0 / p.nd) % p.per;
  }
  return p;
}
// `w0`: the reservation word of the first queue, if the caller has read it (its load then
// overlaps the caller's other loads), else kNoWord
constexpr uint64_t kNoWord = ~0ull;
__device__ __forceinline__ bool sq_reserve_dev(const Dev &d, uint32_t q0, uint32_t dv, uint32_t n, uint32_t &q,
                                               uint32_t &slot, uint32_t &ticket, bool pf = false,
                                               uint64_t w0 = kNoWord) {
  const SqPick p = sq_pick(d, q0, pf);
  // a request made ahead of need tries two queues: when they are full the device is
  // saturated and the request is dropped (a hint), not spread over every queue
  const uint32_t tries = pf ? min(p.per, 2u) : p.per;
  for (uint32_t k = 0; k < tries; ++k) {
    uint32_t kk = p.k0 + k;
    if (kk >= p.per) kk -= p.per;
    uint32_t qq = p.base + kk * p.nd + dv;
    const bool old_word = k == 0 && w0 != kNoWord;
    if (sq_try_reserve(d, qq, n, old_word ? w0 : ld_rlx64(&d.sq_resv[qq]), old_word, slot, ticket)) {
      q = qq;
      return true;
    }
  }
  atomicAdd(stat_ptr(d, S_SQ_FULL), 1ull);
  return false;
}
__device__ __forceinline__ uint64_t sq_first_word(const Dev &d, uint32_t q0, uint32_t dv, bool pf) {
  const SqPick p = sq_pick(d, q0, pf);
  return ld_rlx64(&d.sq_resv[p.base + p.k0 * p.nd + dv]);
}

// The first queue sq_reserve_dev tries for a request of this class holds more than
// 3/4 of its depth in flight: a request made ahead of need is then dropped before it
// claims a line (one load instead of a claim, a failed reservation and an unclaim).
__device__ __forceinline__ bool sq_crowded(const Dev &d, uint32_t q0, uint32_t dv, bool pf) {
  return (uint32_t)(sq_first_word(d, q0, dv, pf) >> 32) > (d.depth - 1) / 4 * 3;
}

// Alg. 2, enqueue_cmd: write the 64-byte command into its reserved slot.  CID = slot index
// (unique while the command is outstanding).  sq_ring, by the same thread, issues it.
__device__ __forceinline__ void sq_write(const Dev &d, uint32_t q, uint32_t slot, uint32_t ticket,
                                         uint32_t opcode, uint64_t prp1, uint64_t page,
                                         uint64_t ctx) {
  uint64_t i = (uint64_t)q * d.depth + slot;
  uint32_t *e = d.sq[i].dw;
  uint64_t slba = block_of_page(d, page) * (kPage / 512);
  // dw2-3 (reserved in NVMe) carry the commit time for the device's trace
  uint64_t now = gtimer();
  int4 a = make_int4((int)(opcode | (slot << 16)), 1, (int)(uint32_t)now, (int)(uint32_t)(now >> 32));  // dw0-3
  int4 b = make_int4(0, 0, (int)(uint32_t)prp1, (int)(uint32_t)(prp1 >> 32));      // dw4-7
  int4 c = make_int4(0, 0, (int)(uint32_t)slba, (int)(uint32_t)(slba >> 32));      // dw8-11
  int4 f = make_int4((int)(kPage / 512 - 1), 0, 0, 0);                             // dw12-15
  st_cg16(e, a);
  st_cg16(e + 4, b);
  st_cg16(e + 8, c);
  st_cg16(e + 12, f);
  st_rlx64(&d.cmd_ctx[i], ctx);
  st_rlx64(&d.sqe_state[i], ((uint64_t)ticket << 2) | SQE_WRITTEN);
}

// Alg. 2, update_SQE + move_SQ_tail + Attempt_SQDB without a lock: issue the `n` commands
// written to consecutive slots from `ticket` on.  The doorbell counts issued commands,
// so it is the tail, and it equals `ticket` once every command before ours is out: then
// one compare-and-swap issues ours.  If it does not, the slots are marked UPDATED and
// the compare-and-swap is tried once more: either it succeeds now, or the thread that
// issues the command before ours finds the mark (both sides put an sc fence between
// their write and their read) and issues ours with its own -- no thread waits for
// another.  A thread so issues its commands and all UPDATED ones right behind them with one
// doorbell each time it moves the tail.  (The doorbell lock this replaces -- lock, tail,
// two state reads, doorbell, unlock, state read -- had a command wait 5.5 us from its
// commit to the device; the compare-and-swap has 3 us, measured on 256 warps of misses.)
static __device__ __forceinline__ void sq_ring(const Dev &d, uint32_t q, uint32_t ticket, uint32_t n = 1) {
  uint32_t *db = &d.sq_db[q];
  unsigned long long *st = &d.sqe_state[(uint64_t)q * d.depth];
  fence_ar();  // the commands (and what the caller wrote before) reach the device with the doorbell
  uint32_t rung = 0;
  if (atomicCAS(db, ticket, ticket + n) != ticket) {
    for (uint32_t k = 0; k < n; ++k)
      st_rlx64(&st[(ticket + k) & d.dmask], ((uint64_t)(ticket + k) << 2) | SQE_UPDATED);
    fence_sc();
    uint32_t from = ticket, old = atomicCAS(db, from, ticket + n);
    // the issuer before us may have seen the first marks and not yet the others
    while (old != from && old - ticket < n) {
      from = old;
      old = atomicCAS(db, from, ticket + n);
    }
    if (old != from) return;
  }
  for (uint32_t t = ticket + n;;) {
    ++rung;
    fence_sc();
    uint32_t m = 0;
    while (m < d.depth && ld_acq64(&st[(t + m) & d.dmask]) == (((uint64_t)(uint32_t)(t + m) << 2) | SQE_UPDATED)) ++m;
    if (!m) break;
    fence_ar();
    if (atomicCAS(db, t, t + m) != t) break;  // their own thread was faster and looks further
    t += m;
  }
  atomicAdd(stat_ptr(d, S_DOORBELLS), (unsigned long long)rung);
}

// Warp-collective reservation for lanes that need one slot each: the lanes with `want` of
// an aligned group of four share one compare-and-swap on their first lane's queue and
// take consecutive slots, and that lane rings for them all (`n` commands from `first` on;
// n = 0 in the others).  Four, not the whole warp: engines take the commands of one queue
// two at a time, a round trip each.  For bursts, where the threads' compare-and-swaps on a
// queue's two words bound its issue (a flush of 8 k lines, 64 a queue: the last command was
// written 192 us after the first, 96 with groups; the few misses of a lookup or a scan are
// slower with it, 3 %).  For one device only (consecutive slots of a queue).
// False for a lane of a group that found no room.
static __device__ __forceinline__ bool sq_reserve_group(const Dev &d, bool want, uint32_t q0, uint32_t &q,
                                                        uint32_t &slot, uint32_t &ticket, uint32_t &first, uint32_t &n) {
  const unsigned l = lane_id(), base = l & ~3u;
  const uint32_t mine = (__ballot_sync(kFull, want) >> base) & 15u;
  const int lead = (int)base + (mine ? __ffs(mine) - 1 : 0);
  bool ok = false;
  n = 0;
  if (want && lead == (int)l) {
    n = __popc(mine);
    ok = sq_reserve_dev(d, q0, 0, n, q, slot, ticket);
  }
  __syncwarp();
  ok = __shfl_sync(kFull, ok, lead);
  q = __shfl_sync(kFull, q, lead);
  first = __shfl_sync(kFull, ticket, lead);
  ticket = first + __popc(mine & ((1u << (l & 3)) - 1));
  slot = ticket & d.dmask;
  if (!ok) n = 0;
  return ok && want;
}

// ================================================================ in-flight share table
// Sec. 3.4.1: page -> request in flight.  Inserting the page is how a thread takes
// ownership of its miss (or write); any other thread that finds it defers and retries.
// A bucket is one 64-bit word of four 16-bit keys (bit 15 = in use), so a single
// compare-and-swap both sees whether the page is there and inserts it, and no two
// threads can insert it into different slots.  page * sh_mul mod 2^sh_bits (an odd
// multiplier: a bijection of the store's page numbers) gives the bucket in its upper bits
// and the key in its lower 15, so equal keys in a bucket are equal pages.
constexpr uint32_t kShKeyBits = 15;
__device__ __forceinline__ uint32_t sh_hash(const Dev &d, uint64_t page, uint64_t &key) {
  uint64_t y = (page * d.sh_mul) & ((1ull << d.sh_bits) - 1);
  key = (y & 0x7FFFu) | 0x8000u;
  return (uint32_t)(y >> kShKeyBits);
}
__device__ __forceinline__ int sh_find(uint64_t word, uint64_t key) {
  int at = -1;
#pragma unroll
  for (int k = 3; k >= 0; --k)
    if (((word >> (16 * k)) & 0xFFFFu) == key) at = k;
  return at;
}
// returns slot index >= 0 when inserted, -1 when the page is already present, -2 when
// the bucket is full (or too contended).  The insertion acquires: what the page's last
// request wrote before it left the table (tag, store) is seen after it.
__device__ __forceinline__ int64_t sh_insert(const Dev &d, uint64_t page) {
  uint64_t key;
  const uint32_t b = sh_hash(d, page, key);
  uint64_t w = 0;  // most buckets are empty
  for (int tries = 0; tries < 8; ++tries) {
    if (sh_find(w, key) >= 0) return -1;
    int k = sh_find(w, 0);
    if (k < 0) return -2;
    uint64_t old = atom_cas_acq(&d.sh_key[b], w, w | (key << (16 * k)));
    if (old == w) return (int64_t)b * 4 + k;
    w = old;
  }
  return -2;
}
// the caller's earlier writes are ordered before the removal by a fence of its own
__device__ __forceinline__ void sh_clear(const Dev &d, uint64_t slot) {
  atomicAnd(&d.sh_key[slot >> 2], ~(0xFFFFull << (16 * (slot & 3))));
}
__device__ __forceinline__ void sh_remove(const Dev &d, uint64_t slot) {
  st_rlx64(&d.sh_val[slot], 0ull);  // the next owner finds it 0
  fence_ar();
  sh_clear(d, slot);
}
// Token of the read in flight for `page`, ~0 when there is none (or it is not
// published yet).  The key is read again after the value: an entry removed (and maybe reused)
// meanwhile is not taken; one re-inserted for the same page carries a token of the same
// page, which is as good.
__device__ __forceinline__ uint64_t sh_token(const Dev &d, uint64_t page) {
  uint64_t key;
  const uint32_t b = sh_hash(d, page, key);
  int k = sh_find(ld_acq64(&d.sh_key[b]), key);
  if (k < 0) return ~0ull;
  uint64_t v = ld_acq64(&d.sh_val[(uint64_t)b * 4 + k]);
  if (v && sh_find(ld_acq64(&d.sh_key[b]), key) == k) return v - 1;
  return ~0ull;
}

// ================================================================ cache (Sec. 3.4)
enum Probe { P_HIT = 0, P_BUSY = 1, P_MISS = 2 };

// Look the page up in its set.  READY/MODIFIED -> hit (case a): the reference bit is
// set and, with `pin`, the line is pinned against eviction.  BUSY -> in flight
// (case c).  Otherwise a miss.
// tags of 8 ways at once: four independent 16-byte loads from L2 (one round trip);
// every 8-byte tag is read as one access
__device__ __forceinline__ void ld_tags8(const unsigned long long *p, uint64_t t[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    asm volatile("ld.global.cg.v2.u64 {%0,%1}, [%2];" : "=l"(t[2 * k]), "=l"(t[2 * k + 1]) : "l"(p + 2 * k) : "memory");
}

// ... as 32-bit halves: {page bits 0-11, pin, wb, ref, state} and {page bits 12-43}
__device__ __forceinline__ void ld_tags8_halves(const unsigned long long *p, uint32_t lo[8], uint32_t hi[8]) {
  static_assert(PAGE_SHIFT == 20, "the upper half holds the page from bit 12 on");
#pragma unroll
  for (int k = 0; k < 4; ++k)
    asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(lo[2 * k]), "=r"(hi[2 * k]), "=r"(lo[2 * k + 1]), "=r"(hi[2 * k + 1]) : "l"(p + 2 * k) : "memory");
}

// The way of an 8-way tag copy that holds `page` READY or MODIFIED (its tag in t), or
// -1; unrolled, so the copy stays in registers.
__device__ __forceinline__ int match_ready8(const uint64_t pre[8], uint64_t page, uint64_t &t) {
  int w = -1;
#pragma unroll
  for (int k = 7; k >= 0; --k) {
    uint64_t st = tag_state(pre[k]);
    if ((st == ST_READY || st == ST_MODIFIED) && tag_page(pre[k]) == page) {
      w = k;
      t = pre[k];
    }
  }
  return w;
}

__device__ __forceinline__ int cache_probe(const Dev &d, uint64_t page, bool pin, uint32_t &line) {
  uint64_t base = (uint64_t)set_of(page, d.sets) * d.ways;
  uint64_t t = 0;
  int wsel = -1;
  if (d.ways == 8) {  // sets of 8 ways are 64-byte aligned: read them at once
    uint32_t lo[8], hi[8], tl = 0;
    ld_tags8_halves(&d.tag[base], lo, hi);
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if ((lo[k] & 3) && hi[k] == (uint32_t)(page >> 12) && lo[k] >> PAGE_SHIFT == ((uint32_t)page & 0xFFFu)) {
        wsel = k;
        tl = lo[k];
      }
    t = tl;  // state and reference bit
  } else {
    for (uint32_t k = 0; k < d.ways && wsel < 0; ++k) {
      uint64_t tk = ld_rlx64(&d.tag[base + k]);
      if (tag_state(tk) != ST_INVALID && tag_page(tk) == page) {
        wsel = (int)k;
        t = tk;
      }
    }
  }
  if (wsel >= 0) {
    const uint32_t w = (uint32_t)wsel;
    uint64_t st = tag_state(t);
    line = (uint32_t)(base + w);
    if (st == ST_BUSY) return P_BUSY;
    if (!pin) {
      if (!(t & TAG_REF)) atomicOr(&d.tag[base + w], TAG_REF);
      return P_HIT;
    }
    uint64_t old = atom_add_acq(&d.tag[base + w], PIN1);  // line data is read after the pin
    uint64_t ost = tag_state(old);
    if (tag_page(old) == page && (ost == ST_READY || ost == ST_MODIFIED)) {
      if (!(old & TAG_REF)) atomicOr(&d.tag[base + w], TAG_REF);
      return P_HIT;
    }
    atomicAdd(&d.tag[base + w], (unsigned long long)(-(int64_t)PIN1));
    return ost == ST_BUSY && tag_page(old) == page ? P_BUSY : P_MISS;
  }
  return P_MISS;
}

__device__ __forceinline__ void cache_unpin(const Dev &d, uint32_t line) {
  atomicAdd(&d.tag[line], (unsigned long long)(-(int64_t)PIN1));
}

// Give up a victim we claimed but could not use (keeps transient pin bits of others).  A
// MODIFIED victim gets its tag back: its page's in-flight entry, held by the caller, has
// kept everyone from reading the page meanwhile.  A clean one has no such entry: another
// thread may have missed on its page and be filling a second way with it, and two valid
// copies lose updates.  Its way is left INVALID.
__device__ __forceinline__ void cache_unclaim(const Dev &d, uint32_t line, uint64_t old_tag) {
  uint64_t cur = ld_rlx64(&d.tag[line]);
  const uint64_t back = tag_state(old_tag) == ST_MODIFIED ? old_tag & ~PIN_MASK : 0;
  for (int i = 0; i < 64; ++i) {
    uint64_t want = back | (cur & PIN_MASK);
    uint64_t got = atomicCAS(&d.tag[line], (unsigned long long)cur, (unsigned long long)want);
    if (got == cur) return;
    cur = got;
  }
}

enum Miss { M_ISSUED = 0, M_HIT = 1, M_BUSY = 2, M_RETRY = 3 };

struct Issued {
  uint32_t q, slot, ticket;  // the command issued last (the read, when there is one)
  int code;  // 1 fill, 2 evict READY, 3 write-back MODIFIED
};

// What one thread's miss holds between cache_claim, cache_reserve and cache_issue: the
// claimed line, its old tag, the in-flight entries of the page and of a MODIFIED victim,
// then the reserved slots.  wb: the victim must be copied to the staging page of
// (q, slot) before cache_issue.  w0: the first queue's reservation word, read beside the claim.
struct Claim {
  uint64_t old, w0;
  int64_t sh, sh_wb;
  uint32_t line, q, slot, ticket;
  bool wb, fill;
};
__device__ __forceinline__ uint8_t *claim_staging(const Dev &d, const Claim &c) {
  return d.staging + ((uint64_t)c.q * d.depth + c.slot) * kPage;
}

// The rare miss whose MODIFIED victim lives on another device than the page that
// replaces it: the write-back takes a demand slot of its device, the read a slot of the
// page's device.  If the read's slot cannot be had, the write-back's slot is spent on a
// no-op command (a reserved slot must be issued) and the miss is retried holding
// nothing.  The write-back is issued here; the read is left to cache_issue.
// Out of line, so that the common miss path stays small.
static __device__ __noinline__ int cache_reserve_split(uint64_t page, uint32_t q0, Claim &c, bool pf) {
  const Dev &d = shared_dev();
  uint32_t wq = 0, wslot = 0, wticket = 0, q = 0, slot = 0, ticket = 0;
  if (!sq_reserve_dev(d, q0, dev_of_page(d, tag_page(c.old)), 1, wq, wslot, wticket, false)) {
    cache_unclaim(d, c.line, c.old);
    sh_remove(d, (uint64_t)c.sh_wb);
    sh_remove(d, (uint64_t)c.sh);
    return M_RETRY;
  }
  if (!sq_reserve_dev(d, q0, dev_of_page(d, page), 1, q, slot, ticket, pf)) {
    sq_write(d, wq, wslot, wticket, OP_FLUSH, 0, 0, ctx_make(CTX_NOP, 0, 0));
    cache_unclaim(d, c.line, c.old);
    sh_remove(d, (uint64_t)c.sh_wb);
    sh_remove(d, (uint64_t)c.sh);
    sq_ring(d, wq, wticket);
    return M_RETRY;
  }
  uint8_t *stg = d.staging + ((uint64_t)wq * d.depth + wslot) * kPage;
  fence_ar();  // the line is read after it was claimed
  lane_copy_page(stg, line_ptr(d, c.line));
  sq_write(d, wq, wslot, wticket, OP_WRITE, (uint64_t)stg, tag_page(c.old), ctx_make(CTX_WB, (uint32_t)c.sh_wb, 0));
  atomicAdd(stat_ptr(d, S_WRITEBACKS), 1ull);
  sq_ring(d, wq, wticket);
  c.q = q;
  c.slot = slot;
  c.ticket = ticket;
  c.wb = false;  // already on its way
  return M_ISSUED;
}

// Victim search of a miss in `set` (Sec. 3.4 cases (b) and (d)): the lowest way with
// an INVALID, unpinned tag, else the clock sweep from the set's hand (a way whose
// reference bit is set has it cleared and is passed; BUSY, pinned and written-back
// ways are passed; under FIFO no bit is looked at).  The chosen way is claimed by
// compare-and-swap from the tag that was read, as BUSY for the new page (`claimed`).
// Returns the way (old = its tag before, 0 when it was INVALID; sh_wb = the Share Table
// entry of the write-back of a MODIFIED victim) or -1.
//
// pick_victim8, sets of 8 ways: the sweep is done on the copy of the tags that the
// caller has just read, as bit masks over the ways in the hand's order and without
// branches, so that a claim costs one round trip after that read (hand and cleared
// reference bits are updated without waiting).  A claim that fails (the way was taken or
// touched meanwhile) passes the way.  pick_victim reads every way when the sweep gets to
// it, two round trips a step.
static __device__ __forceinline__ int pick_victim8(const Dev &d, uint32_t set, const uint32_t (&lo)[8],
                                                   const uint32_t (&hi)[8], uint32_t hand, uint64_t claimed,
                                                   uint64_t &old, int64_t &sh_wb) {
  unsigned long long *tags = &d.tag[(uint64_t)set * 8];
  uint32_t zero = 0, skip = 0, ref = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    zero |= ((lo[w] | hi[w]) == 0 ? 1u : 0u) << w;
    skip |= ((lo[w] & (uint32_t)(PIN_MASK | TAG_WB)) != 0 || (lo[w] & 3) == ST_BUSY ? 1u : 0u) << w;
    ref |= (lo[w] & 3 ? (lo[w] >> 2) & 1u : 0u) << w;
  }
  if (d.policy != kPolicyClock) ref = 0;
  const uint32_t h0 = hand & 7;
  uint32_t rskip = ((skip * 0x101u) >> h0) & 0xFF, rref = ((ref * 0x101u) >> h0) & 0xFF, passed = 0;
  for (;;) {
    // an INVALID way, else the first way the hand finds unreferenced, else (second turn)
    // the first one whose bit the first turn has cleared
    const uint32_t first = ~rskip & ~rref & ~passed & 0xFF, second = (rref | passed) & ~rskip;
    if (!(zero | first | second)) {
      atomicAdd(&d.hand[set], 17u);
      return -1;
    }
    const uint32_t p = __ffs(first ? first : second) - 1;
    const uint32_t w = zero ? __ffs(zero) - 1 : (h0 + p) & 7;
    uint32_t clear = zero ? 0 : (first ? rref & ~rskip & ((1u << p) - 1) : rref & ~rskip);
    passed |= clear;
    rref &= ~clear;
    clear = ((clear * 0x101u) >> (8 - h0)) & 0xFF;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if ((clear >> k) & 1u) atomicAnd(&tags[k], ~TAG_REF);
    uint32_t tl = 0, th = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k == (int)w) {
        tl = lo[k];
        th = hi[k];
      }
    if (!zero && (passed >> p & 1u)) tl &= ~(uint32_t)TAG_REF;
    const uint64_t tw = (uint64_t)th << 32 | tl;
    if ((tl & 3) == ST_MODIFIED) sh_wb = sh_insert(d, tag_page(tw));
    if (((tl & 3) != ST_MODIFIED || sh_wb >= 0) &&
        atomicCAS(&tags[w], (unsigned long long)tw, (unsigned long long)claimed) == tw) {
      if (!zero) atomicAdd(&d.hand[set], (first ? 0u : 8u) + p + 1);
      old = (tl & 3) == ST_INVALID ? 0 : tw;
      return (int)w;
    }
    if (sh_wb >= 0) sh_remove(d, (uint64_t)sh_wb);
    sh_wb = -1;
    zero &= zero - 1;  // (0 stays 0)
    rskip |= 1u << ((w - h0) & 7);
  }
}
static __device__ __noinline__ int64_t pick_victim(uint32_t set, uint64_t claimed, uint64_t &old, int64_t &sh_wb) {
  const Dev &d = shared_dev();
  const uint32_t ways = d.ways;
  const uint64_t base = (uint64_t)set * ways;
  for (uint32_t w = 0; w < ways; ++w) {
    uint64_t t = ld_rlx64(&d.tag[base + w]);
    if (t == 0 && atomicCAS(&d.tag[base + w], 0ull, (unsigned long long)claimed) == 0ull) {
      old = 0;
      return w;
    }
  }
  for (uint32_t step = 0; step < 2 * ways + 1; ++step) {
    uint32_t w = atomicAdd(&d.hand[set], 1u) % ways;
    uint64_t t = ld_rlx64(&d.tag[base + w]);
    uint64_t st = tag_state(t);
    if (st == ST_INVALID) {
      if ((t & PIN_MASK) == 0 && atomicCAS(&d.tag[base + w], (unsigned long long)t, (unsigned long long)claimed) == t) {
        old = 0;
        return w;
      }
      continue;
    }
    if (st == ST_BUSY || (t & (PIN_MASK | TAG_WB))) continue;
    if (d.policy == kPolicyClock && (t & TAG_REF)) {
      atomicAnd(&d.tag[base + w], ~TAG_REF);
      continue;
    }
    if (st == ST_MODIFIED) {
      sh_wb = sh_insert(d, tag_page(t));
      if (sh_wb < 0) continue;
    }
    if (atomicCAS(&d.tag[base + w], (unsigned long long)t, (unsigned long long)claimed) == t) {
      old = t;
      return w;
    }
    if (sh_wb >= 0) {
      sh_remove(d, (uint64_t)sh_wb);
      sh_wb = -1;
    }
  }
  return -1;
}

// Cases (b) and (d) for one thread, first part: take ownership of the page's miss in the
// share table, probe once more (the page may have come in meanwhile), pick and claim a
// way.  Nothing in the three parts waits: on any shortage every claim is undone and M_RETRY
// returned.  The chain of dependent L2 round trips bounds a miss (not bandwidth):
// in-flight entry, set and hand, claim, reservation, doorbell -- the first queue's
// reservation word is loaded beside the in-flight entry.
//
// fill=false (writes of whole pages): the caller already owns the page's share entry
// `sh_own`; the way is claimed BUSY without a read, the caller writes the line and
// publishes it.  A MODIFIED victim is still written back first.
static __device__ __forceinline__ int cache_claim(const Dev &d, uint64_t page, uint32_t q0, Claim &c, bool fill = true,
                                               int64_t sh_own = -1, bool pf = false) {
  c.sh = sh_own;
  c.sh_wb = -1;
  c.old = 0;
  c.wb = false;
  c.fill = fill;
  c.q = 0xFFFFFFFFu;
  c.slot = c.ticket = 0;
  c.w0 = kNoWord;
  if (fill) {
    c.w0 = sq_first_word(d, q0, dev_of_page(d, page), pf);
    c.sh = sh_insert(d, page);
    if (c.sh < 0) {
      // another thread is at the page (a request made without waiting is done with it) or
      // the bucket is full
      atomicAdd(stat_ptr(d, S_SHARE_RETRIES), 1ull);
      c.line = 0;
      return c.sh == -1 ? M_BUSY : M_RETRY;
    }
  }
  const uint32_t set = set_of(page, d.sets);
  const uint64_t base = (uint64_t)set * d.ways, claimed = tag_make(page, ST_BUSY, true);
  int64_t victim = -1;
  int there = -1;  // way that holds the page already
  uint64_t tw = 0;
  if (d.ways == 8) {
    uint32_t lo[8], hi[8];
    const uint32_t hand = ld_rlx32(&d.hand[set]);
    ld_tags8_halves(&d.tag[base], lo, hi);
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if ((lo[k] & 3) && hi[k] == (uint32_t)(page >> 12) && lo[k] >> PAGE_SHIFT == ((uint32_t)page & 0xFFFu)) {
        there = k;
        tw = lo[k];
      }
    if (there < 0) victim = pick_victim8(d, set, lo, hi, hand, claimed, c.old, c.sh_wb);
  } else {
    for (uint32_t k = 0; k < d.ways && there < 0; ++k) {
      tw = ld_rlx64(&d.tag[base + k]);
      if (tag_state(tw) != ST_INVALID && tag_page(tw) == page) there = (int)k;
    }
    if (there < 0) victim = pick_victim(set, claimed, c.old, c.sh_wb);
  }
  if (there >= 0) {
    c.line = (uint32_t)(base + there);
    if (fill) sh_remove(d, (uint64_t)c.sh);
    if (tag_state(tw) == ST_BUSY) return M_BUSY;
    if (!(tw & TAG_REF)) atomicOr(&d.tag[c.line], TAG_REF);
    return M_HIT;
  }
  if (victim < 0) {
    if (fill) sh_remove(d, (uint64_t)c.sh);
    atomicAdd(stat_ptr(d, S_EAGAIN), 1ull);
    return M_RETRY;
  }
  c.line = (uint32_t)(base + victim);
  c.wb = tag_state(c.old) == ST_MODIFIED;
  return M_ISSUED;
}

// Second part: reserve queue slots, right before the commands are written and issued: a
// queue's commands reach the device in the order of their slots, so a slot held while
// other lanes of the warp still look for lines would hold up every other warp's commands
// behind it (reserved with the claim, a twentieth of the commands of a page-read burst
// waited 100 us).
static __device__ __forceinline__ int cache_reserve(const Dev &d, uint64_t page, uint32_t q0, Claim &c, bool pf) {
  if (c.wb && c.fill && d.ndev > 1 && dev_of_page(d, tag_page(c.old)) != dev_of_page(d, page))
    return cache_reserve_split(page, q0, c, pf);
  // a write-back and its refill take two consecutive slots of one queue of their
  // device, reserved together (a write-back rides in the demand class: a fill waits
  // behind it)
  const uint32_t nslots = (c.wb ? 1u : 0u) + (c.fill ? 1u : 0u);
  if (nslots && !sq_reserve_dev(d, q0, dev_of_page(d, c.wb ? tag_page(c.old) : page), nslots, c.q, c.slot, c.ticket,
                                pf && !c.wb, c.wb ? kNoWord : c.w0)) {
    cache_unclaim(d, c.line, c.old);
    if (c.wb) sh_remove(d, (uint64_t)c.sh_wb);
    if (c.fill) sh_remove(d, (uint64_t)c.sh);
    return M_RETRY;
  }
  if (c.wb) fence_ar();  // the line is read after it was claimed
  return M_ISSUED;
}

// Third part: write the commands of a claim (a MODIFIED victim's page is in its staging
// page by now) and issue them.
static __device__ __forceinline__ void cache_issue(const Dev &d, uint64_t page, const Claim &c, Issued &is) {
  is.q = c.q;
  is.slot = c.slot;
  is.ticket = c.ticket;
  is.code = tag_state(c.old) == ST_MODIFIED ? 3 : (c.old ? 2 : 1);
  if (c.old) atomicAdd(stat_ptr(d, S_EVICTIONS), 1ull);
  if (c.wb) {
    sq_write(d, c.q, c.slot, c.ticket, OP_WRITE, (uint64_t)claim_staging(d, c), tag_page(c.old),
             ctx_make(CTX_WB, (uint32_t)c.sh_wb, 0));
    atomicAdd(stat_ptr(d, S_WRITEBACKS), 1ull);
  }
  if (c.fill) {
    if (c.wb) {
      is.slot = (c.slot + 1) & d.dmask;
      is.ticket = c.ticket + 1;
    }
    // the read's token + 1 (0 = none yet), for threads that find the page in flight
    // (Sec. 3.4 case (c)); the doorbell's fence publishes it
    st_rlx64(&d.sh_val[c.sh], (((uint64_t)c.q << 48) | ((uint64_t)is.slot << 32) | is.ticket) + 1);
    sq_write(d, c.q, is.slot, is.ticket, OP_READ, (uint64_t)line_ptr(d, c.line), page,
             ctx_make(CTX_FILL, (uint32_t)c.sh, c.line));
    atomicAdd(stat_ptr(d, S_MISSES), 1ull);
  }
  const uint32_t n = (c.wb ? 1u : 0u) + (c.fill ? 1u : 0u);
  if (n) sq_ring(d, c.q, c.ticket, n);
}

// all three for a lane on its own
static __device__ __noinline__ int cache_miss_call(uint64_t page, uint32_t q0, uint32_t &line, Issued &is, bool fill,
                                                   int64_t sh_own, bool pf) {
  const Dev &d = shared_dev();
  Claim c;
  int m = cache_claim(d, page, q0, c, fill, sh_own, pf);
  if (m == M_ISSUED) m = cache_reserve(d, page, q0, c, pf);
  if (m != M_RETRY) line = c.line;
  if (m != M_ISSUED) return m;
  if (c.wb) lane_copy_page(claim_staging(d, c), line_ptr(d, c.line));
  cache_issue(d, page, c, is);
  return M_ISSUED;
}
static __device__ __forceinline__ int cache_miss(const Dev &, uint64_t page, uint32_t q0, uint32_t &line, Issued &is,
                                                 bool fill = true, int64_t sh_own = -1, bool pf = false) {
  return cache_miss_call(page, q0, line, is, fill, sh_own, pf);
}

__device__ __forceinline__ uint64_t make_token(uint32_t q, uint32_t slot, uint32_t ticket) {
  return ((uint64_t)q << 48) | ((uint64_t)slot << 32) | ticket;
}

// ---------------------------------------------------------------- warp-level requests
// Sec. 3.3.2 two-level coalescing: lanes asking for the same page are matched with
// __match_any_sync and only the lowest lane of each group goes to the cache.
//
// warp_request: every lane with `want` names a page.  Leaders probe; misses are issued
// (one doorbell per queue per warp).  With wait=false this is a prefetch: the call
// returns once every page is READY, in flight or could not be started.  With
// wait=true it returns once every page is READY (no pins are held while waiting).
// Returns false on timeout/abort.  `tok` (leaders) receives the token of the read the
// lane itself issued, AGILE_TOKEN_HIT otherwise.
// `outcome` (optional) receives, in every lane, bit 0: this call sent a read to the
// device (a page READY or already in flight adds nothing); bit 1: some hint was
// dropped because the device is saturated.
// `pf`: the pages are requested ahead of need (prefetch queues, served after demand).
// `limit`: how many misses a hint may send.
// `hint`: a speculative request of an application's lookahead, dropped (no retry) when
// its first queue is crowded or no queue has room -- the device is saturated.
// Out of line: one copy per kernel keeps the applications' loops and the instruction
// cache footprint small (with five inlined copies a lookup kernel's warps waited 9 of 24
// cycles between instructions for instruction fetches); a call costs little next to the
// round trips of a request.
struct Requested {
  uint64_t tok;
  uint32_t outcome;  // bit 0 sent, bit 1 dropped, bit 2 ok; code in the upper half
};
static __device__ __noinline__ Requested warp_request_body(bool want, uint64_t page, uint32_t q0, bool wait,
                                                           uint64_t deadline, bool pf, bool hint, uint32_t limit) {
  const Dev &d = shared_dev();
  uint64_t tok = ~0ull;
  int code = 0;
  unsigned grp = __match_any_sync(kFull, want ? page : ~0ull);
  int lead_lane = __ffs(grp) - 1;
  bool leader = want && lead_lane == (int)lane_id();
  stat_warp(d, S_WARP_COALESCED, (want && !leader) ? 1u : 0u);
  bool need = leader;
  uint32_t line = 0;
  bool ok = true;
  bool first = true;
  uint32_t ns = 32;
  uint32_t retries = 0;
  bool dropped = false, sent = false;
  while (__any_sync(kFull, need)) {
    int m = M_RETRY;
    bool missed = false;
    Claim c;
    c.wb = false;
    if (need) {
      int pr = cache_probe(d, page, false, line);
      if (pr == P_HIT) {
        need = false;
        if (first) atomicAdd(stat_ptr(d, S_HITS), 1ull);
      } else if (pr == P_BUSY) {
        if (first) atomicAdd(stat_ptr(d, S_BUSY_HITS), 1ull);
        if (!wait) need = false;
      } else {
        missed = true;
      }
    }
    if (hint) {
      // beyond `limit` misses, or with the device saturated, a hint is dropped
      const unsigned away = __ballot_sync(kFull, missed);
      if (missed && !wait &&
          ((uint32_t)__popc(away & ((1u << lane_id()) - 1)) >= limit || sq_crowded(d, q0, dev_of_page(d, page), pf))) {
        missed = need = false;
        dropped = true;
      }
    }
    if (__any_sync(kFull, missed)) {
      if (missed) {
        m = cache_claim(d, page, q0, c, true, -1, pf);
        if (m != M_RETRY) line = c.line;
      }
      __syncwarp();
      if (m == M_ISSUED) m = cache_reserve(d, page, q0, c, pf);
      // MODIFIED victims are copied to their staging pages by the whole warp: its reads come
      // after the claiming lane's fence (votes and shuffles order no memory)
      __syncwarp();
      for (unsigned wb = __ballot_sync(kFull, m == M_ISSUED && c.wb); wb; wb &= wb - 1) {
        const int j = __ffs(wb) - 1;
        const uint64_t src = __shfl_sync(kFull, (uint64_t)line_ptr(d, c.line), j);
        const uint64_t dst = __shfl_sync(kFull, (uint64_t)claim_staging(d, c), j);
        warp_copy_page((void *)dst, (const void *)src);
      }
      __syncwarp();
      if (missed) {
        if (m == M_ISSUED) {
          Issued is;
          cache_issue(d, page, c, is);
          sent = true;
          tok = ((uint64_t)is.q << 48) | ((uint64_t)is.slot << 32) | is.ticket;
          code = is.code;
          if (!wait) need = false;
        } else if (m == M_HIT) {
          need = false;
        } else if (m == M_BUSY) {
          if (!wait) need = false;
        } else if (!wait && (hint || ++retries >= 4)) {
          need = false;  // a prefetch is a hint: give up when nothing can be evicted now
          if (hint) dropped = true;
        }
      }
      __syncwarp();
    }
    first = false;
    if (__any_sync(kFull, need)) {
      if (need) {
        if (gtimer() > deadline || aborted(d)) {
          set_error(d, -110);
          need = false;
          ok = false;
        } else {
          // wait for the in-flight line without holding anything, then probe again
          // (short sleeps: a fill completes within microseconds)
          backoff(ns, 256);
        }
      }
    }
  }
  uint32_t outcome = (__any_sync(kFull, sent) ? 1u : 0u) | (__any_sync(kFull, dropped) ? 2u : 0u) |
                     (__all_sync(kFull, ok) ? 4u : 0u);
  return Requested{tok, outcome | (uint32_t)code << 16};
}
static __device__ __forceinline__ bool warp_request(const Dev &, bool want, uint64_t page, uint32_t q0, bool wait,
                                                    uint64_t deadline, uint64_t *tok = nullptr, int *code = nullptr,
                                                    uint32_t *outcome = nullptr, bool pf = false, bool hint = false,
                                                    uint32_t limit = 32) {
  const Requested r = warp_request_body(want, page, q0, wait, deadline, pf, hint, limit);
  if (tok) *tok = r.tok;
  if (code) *code = (int)(r.outcome >> 16);
  if (outcome) *outcome = r.outcome & 3u;
  return (r.outcome & 4u) != 0;
}

// Warp-cooperative probe of one page (uniform across the warp): lane w < ways loads
// the tag of way w, so the whole set is read in one round trip; on a READY/MODIFIED
// match the matching lane pins the line.  Same outcome as cache_probe(pin=true).
__device__ __forceinline__ int warp_probe_pin(const Dev &d, uint64_t page, uint32_t &line) {
  unsigned l = lane_id();
  uint64_t base = (uint64_t)set_of(page, d.sets) * d.ways;
  uint64_t t = l < d.ways ? ld_rlx64(&d.tag[base + l]) : 0;
  bool match = l < d.ways && tag_state(t) != ST_INVALID && tag_page(t) == page;
  unsigned m = __ballot_sync(kFull, match);
  if (!m) return P_MISS;
  int w = __ffs(m) - 1;
  line = (uint32_t)(base + w);
  int pr = P_MISS;
  if ((int)l == w) {
    if (tag_state(t) == ST_BUSY) {
      pr = P_BUSY;
    } else {
      uint64_t old = atom_add_acq(&d.tag[line], PIN1);  // line data is read after the pin
      uint64_t ost = tag_state(old);
      if (tag_page(old) == page && (ost == ST_READY || ost == ST_MODIFIED)) {
        if (!(old & TAG_REF)) atomicOr(&d.tag[line], TAG_REF);
        pr = P_HIT;
      } else {
        atomicAdd(&d.tag[line], (unsigned long long)(-(int64_t)PIN1));
        pr = (ost == ST_BUSY && tag_page(old) == page) ? P_BUSY : P_MISS;
      }
    }
  }
  __syncwarp();  // the pin's acquire comes before every lane's reads of the line
  return __shfl_sync(kFull, pr, w);
}

// warp_request without its optional results
static __device__ __forceinline__ bool warp_request_call(const Dev &d, bool want, uint64_t page, uint32_t q0,
                                                         bool wait, uint64_t deadline, bool pf = false) {
  return warp_request(d, want, page, q0, wait, deadline, nullptr, nullptr, nullptr, pf);
}

// The warp needs one page pinned (uniform `page`): probe with a pin; on a miss the warp
// issues the read and, holding nothing, watches the line's tag until the fill is there,
// then probes again.  Returns the line in every lane, or false on timeout/abort.  The
// caller unpins it (one unpin per pin).
constexpr uint32_t kNoLine = 0xFFFFFFFFu;
static __device__ __noinline__ uint32_t warp_pin_page_body(uint64_t page, uint32_t q0, uint64_t deadline) {
  const Dev &d = shared_dev();
  uint32_t ns = 32;
  for (int round = 0;; ++round) {
    uint32_t line = 0;
    int pr = warp_probe_pin(d, page, line);
    if (pr == P_HIT) {
      if (lane_id() == 0 && round == 0) atomicAdd(stat_ptr(d, S_HITS), 1ull);
      return line;
    }
    if (pr == P_BUSY) {
      if (lane_id() == 0) {
        if (round == 0) atomicAdd(stat_ptr(d, S_BUSY_HITS), 1ull);
        for (uint32_t spin = 0;; ++spin) {
          uint64_t t = ld_rlx64(&d.tag[line]);
          if (tag_page(t) != page || tag_state(t) != ST_BUSY) break;
          if ((spin & 7) == 7 && (gtimer() > deadline || aborted(d))) break;
          __nanosleep(32);
        }
      }
      __syncwarp();
    } else {
      uint32_t outcome = 0;
      if (!warp_request(d, lane_id() == 0, page, q0, false, deadline, nullptr, nullptr, &outcome)) return kNoLine;
      // nothing sent: no way could be evicted, or another warp is at the page.  With every way
      // of the set in flight a warp that claims again at once takes the next page that
      // arrives, before the warp that waits for it has pinned it, and that warp reads it
      // again: at a cap of 256 ns (SSD-like device, 2^20 vertices, cache 1/16) a BFS took
      // 53-139 ms sync and 108 async, at 2, 4, 8 and 16 us 35, 26, 25 and 25 (34, 27, 27, 27).
      if (!(outcome & 1u)) backoff(ns, 8192);
    }
    if (aborted(d)) return kNoLine;
    if (gtimer() > deadline) {
      if (lane_id() == 0) set_error(d, -110);
      return kNoLine;
    }
  }
}
static __device__ __forceinline__ bool warp_pin_page(const Dev &, uint64_t page, uint32_t q0, uint64_t deadline,
                                                     uint32_t &line_out) {
  line_out = warp_pin_page_body(page, q0, deadline);
  return line_out != kNoLine;
}

// Asynchronous requests ahead of use pay a probe per page even when they have nothing
// to do: every page already resident or in flight, or the device saturated (the hints
// are dropped).
// A warp whose lookahead keeps finding nothing to do requests less often: after such a
// round it skips the next `span` rounds (span 1, 3, 7, ... up to 63).  A round that
// sends work to the device brings it back to every round, and so does a miss met later
// by the warp's own gather -- unless the last round was dropped for saturation (the
// gather misses then because the hints were dropped, and more lookahead would only be
// dropped again).  Skipped pages are fetched when used, as in synchronous mode.
struct Backoff {
  uint32_t skip = 0, span = 0;
  bool sat = false;
  __device__ __forceinline__ bool take() {  // true: request this round
    if (skip) {
      --skip;
      return false;
    }
    return true;
  }
  // outcome of warp_request: bit 0 work sent to the device, bit 1 hints dropped
  __device__ __forceinline__ void result(uint32_t outcome) {
    if (outcome & 1u) {
      span = 0;
      sat = false;
    } else {
      span = span < 63 ? 2 * span + 1 : 63;
      skip = span;
      sat = (outcome & 2u) != 0;
    }
  }
  __device__ __forceinline__ void missed() {
    if (!sat) skip = span = 0;
  }
};

// what an application warp knows about its launch
struct AppCtx {
  uint32_t warp;     // app warp index in [0, n_warps)
  uint32_t n_warps;  // app warps in the grid
  uint32_t q0;       // this lane's home queue (Sec. 3.3.1: by thread index)
  uint64_t deadline;
};

// Requests a warp takes at a time when `warps` warps share `n`: enough for all of them, a
// multiple of `part`, at most 32.
__host__ __device__ constexpr uint32_t requests_a_step(uint64_t n, uint32_t warps, uint32_t part) {
  const uint64_t each = (n + warps - 1) / warps, parts = (each + part - 1) / part;
  return parts < 32 / part ? (uint32_t)parts * part : 32 / part * part;
}

// ================================================================ user kernel API
// The device side of Listing 1 (Sec. 3.5) for kernels that run inside a library launch
// (agile_device.cuh launches them): a warp's lanes issue reads, continue with other
// work, test or wait for each read's token, then copy the page.  No call here waits
// while it holds a cache line or a queue slot.

// Token state (agile_test): 0 done, AGILE_EIO done with an error, 1 still in flight.
__device__ __forceinline__ int token_state(const Dev &d, uint64_t tok) {
  if (tok == ~0ull) return 0;
  uint32_t q = (uint32_t)(tok >> 48), slot = (uint32_t)(tok >> 32) & 0xFFFFu, ticket = (uint32_t)tok;
  if (q >= d.Q || slot >= d.depth) return -22;
  uint64_t w = ld_acq64(&d.cmpl[(uint64_t)q * d.depth + slot]);
  uint32_t wt = (uint32_t)(w >> 32);
  if (!(w & 1) || (int32_t)(wt - ticket) < 0) return 1;
  // a later command of the slot has completed: this one completed before it
  if (wt == ticket && ((w >> 1) & 0x7FFF) != 0) return -5;
  return 0;
}

// asyncRead, issue part (warp-collective): lanes with `want` request `page`.  The
// pages of equal requests are merged (the lowest lane goes to the cache); nothing waits
// for data.  Returns the lane's token: AGILE_TOKEN_HIT (~0) when the page was READY,
// else the token of the read that fills it -- issued here, or found in flight (the
// share table names it).  ~0 too after a deadline or an abort (the data is then fetched
// by agile_copy_page).
static __device__ uint64_t api_issue_read(const Dev &d, const AppCtx &a, bool want, uint64_t page) {
  unsigned grp = __match_any_sync(kFull, want ? page : ~0ull);
  int lead = __ffs(grp) - 1;
  bool leader = want && lead == (int)lane_id();
  uint64_t tok = ~0ull;
  bool need = leader;
  uint32_t ns = 64;
  while (__any_sync(kFull, need)) {
    if (need) {
      uint32_t line = 0;
      Issued is{};
      int pr = cache_probe(d, page, false, line);
      if (pr == P_HIT) {
        need = false;
      } else if (pr == P_BUSY) {
        uint64_t t = sh_token(d, page);
        if (t != ~0ull) {
          tok = t;
          need = false;
        }
      } else {
        int m = cache_miss(d, page, a.q0, line, is);
        if (m == M_ISSUED) {
          tok = make_token(is.q, is.slot, is.ticket);
          need = false;
        } else if (m == M_HIT) {
          need = false;
        }
      }
      if (need && (gtimer() > a.deadline || aborted(d))) need = false;
    }
    if (__any_sync(kFull, need)) backoff(ns, 1024);
  }
  tok = __shfl_sync(kFull, tok, lead & 31);
  return want ? tok : ~0ull;
}

// agile_test: non-blocking ("continue" while it is 1)
__device__ __forceinline__ int api_test(const Dev &d, uint64_t tok) { return token_state(d, tok); }

// agile_wait: the transaction barrier of Sec. 3.2.1 for one token, bounded: 0 done,
// AGILE_EIO done with an error, AGILE_ETIMEDOUT when `deadline_ns` (%globaltimer) passes
// first.  The caller holds no pin while it waits (the library never does); a timeout
// is returned to the caller and recorded nowhere else.
__device__ __forceinline__ int api_wait(const Dev &d, uint64_t tok, uint64_t deadline_ns) {
  uint32_t ns = 64;
  for (;;) {
    int st = token_state(d, tok);
    if (st != 1) return st;
    if (gtimer() > deadline_ns) return -110;
    backoff(ns, 1024);
  }
}

// Copy a page (uniform across the warp) from its cache line into dst (4096 bytes,
// 16-byte aligned), with the line pinned for the copy only; a page evicted since its
// read completed is requested again.  False on a timeout of the launch.
static __device__ bool api_copy_page(const Dev &d, const AppCtx &a, uint64_t page, void *dst) {
  uint32_t line;
  if (!warp_pin_page(d, page, a.q0, a.deadline, line)) return false;
  warp_copy_page(dst, line_ptr(d, line));
  __syncwarp();
  if (lane_id() == 0) cache_unpin(d, line);
  return true;
}

// get_row (the synchronous read of part of a page, warp-collective, uniform arguments):
// copy bytes [off, off + nbytes) of `page` to dst, the line pinned for the copy only.
// off, nbytes and dst must be 4-byte aligned and off + nbytes at most one page; else
// AGILE_EINVAL is recorded and false returned.  False also if the launch timed out.
static __device__ bool api_get_row(const Dev &d, const AppCtx &a, uint64_t page, uint32_t off, uint32_t nbytes,
                                   void *dst) {
  if (((off | nbytes | (uint32_t)(uintptr_t)dst) & 3u) || nbytes > kPage || off > kPage - nbytes) {
    if (lane_id() == 0) set_error(d, AGILE_EINVAL);
    return false;
  }
  uint32_t line;
  if (!warp_pin_page(d, page, a.q0, a.deadline, line)) return false;
  const uint8_t *src = line_ptr(d, line) + off;
  int32_t *o = (int32_t *)dst;
  for (uint32_t i = lane_id(); i < nbytes / 4; i += 32) o[i] = ld_cg_s32(src + 4 * i);
  __syncwarp();
  if (lane_id() == 0) cache_unpin(d, line);
  return true;
}

// prefetch (Listing 1 Method-1): start filling the pages of the lanes with `want`.
static __device__ bool api_prefetch(const Dev &d, const AppCtx &a, bool want, uint64_t page) {
  return warp_request_call(d, want, page, a.q0, false, a.deadline, true);
}

// Add rows [j0, j0 + k) (lane j holds row j's line `line_j` and byte offset `off`) to acc
// in increasing j, with several rows' loads in flight at once.
template <int MF4>
__device__ __forceinline__ void sum_rows(const Dev &d, uint32_t j0, uint32_t k, uint32_t line, uint32_t off,
                                         uint32_t nf4, float4 (&acc)[MF4]) {
  unsigned l = lane_id();
  constexpr int RB = MF4 >= 8 ? 1 : 8 / MF4;  // rows in flight: RB * MF4 float4 per lane
  for (uint32_t jb = 0; jb < k; jb += RB) {
    float4 v[RB][MF4];
#pragma unroll
    for (int jj = 0; jj < RB; ++jj) {
      uint32_t j = j0 + jb + jj;
      uint32_t lj = __shfl_sync(kFull, line, j & 31);
      uint32_t oj = __shfl_sync(kFull, off, j & 31);
      const uint8_t *rowp = line_ptr(d, lj) + oj;
#pragma unroll
      for (int c = 0; c < MF4; ++c) {
        uint32_t col = l + 32 * c;
        v[jj][c] = (jb + jj < k && col < nf4) ? ld_cg_f4(rowp + 16 * col) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int jj = 0; jj < RB; ++jj) {
      if (jb + jj < k) {
#pragma unroll
        for (int c = 0; c < MF4; ++c) {
          acc[c].x = __fadd_rn(acc[c].x, v[jj][c].x);
          acc[c].y = __fadd_rn(acc[c].y, v[jj][c].y);
          acc[c].z = __fadd_rn(acc[c].z, v[jj][c].z);
          acc[c].w = __fadd_rn(acc[c].w, v[jj][c].w);
        }
      }
    }
  }
}

// Sum-pool rows 0..cnt-1 into acc, added in increasing lane order (lane j holds row
// j's page `pg` and byte offset `off`).  Lane l adds the float4 columns l, l+32, ... (MF4
// of them, dim/4 in total).
// Each round probes the distinct pages of the rows not yet added, without pinning.  Of
// those not READY, the first `window` ones that nobody has requested are requested
// without waiting (the window keeps what all running warps have requested and not yet
// used within the cache and the queues; rows that hit do not count, so that a bag of
// mostly resident rows is one or two rounds).  Then the pages of the leading run of READY rows are
// pinned, the run is added and every pin let go.  When the next row's page is not READY
// the warp waits for and pins that one page (nothing else pinned meanwhile, Sec. 2.3.2)
// and adds its row: every round adds at least one row, whatever the set conflicts.
// `missed` (optional) is set in every lane when some page had to be requested.
template <int MF4>
static __device__ bool gather_sum(const Dev &d, const AppCtx &a, uint32_t cnt, uint64_t pg, uint32_t off, uint32_t nf4,
                                  float4 (&acc)[MF4], uint32_t window, bool *missed = nullptr) {
  unsigned l = lane_id();
  uint32_t j0 = 0;
  bool first = true;
  const unsigned grp = __match_any_sync(kFull, l < cnt ? pg : ~0ull);
  while (j0 < cnt) {
    bool act = l >= j0 && l < cnt;
    int lead_lane = __ffs(grp & (~0u << j0)) - 1;  // lowest lane of the page not yet added
    bool leader = act && lead_lane == (int)l;
    if (first) stat_warp(d, S_WARP_COALESCED, (act && !leader) ? 1u : 0u);
    uint32_t line = 0;
    int pr = P_HIT;
    if (leader) pr = cache_probe(d, pg, false, line);
    if (first) {
      stat_warp(d, S_HITS, (leader && pr == P_HIT) ? 1u : 0u);
      stat_warp(d, S_BUSY_HITS, (leader && pr == P_BUSY) ? 1u : 0u);
    }
    first = false;
    const unsigned away = __ballot_sync(kFull, leader && pr != P_HIT);
    const bool ask = leader && pr == P_MISS && (uint32_t)__popc(away & ((1u << l) - 1)) < window;
    // a request costs the warp the same few microseconds for one page as for many: the
    // window is refilled when half of it has come in, or the next row needs it
    const unsigned flying = __ballot_sync(kFull, leader && pr == P_BUSY);
    const bool refill = 2 * (uint32_t)__popc(flying) < window || (away & -away & ~flying);
    if (__any_sync(kFull, ask) && refill) {
      if (missed) *missed = true;
      if (!warp_request(d, ask, pg, a.q0, false, a.deadline)) return false;
    }
    // the leading run: its leaders pin
    unsigned hm = __ballot_sync(kFull, act && !((away >> (lead_lane & 31)) & 1u));
    unsigned run = ~(hm >> j0);
    uint32_t k = run ? (uint32_t)(__ffs(run) - 1) : 32u;
    k = min(k, cnt - j0);
    if (k) {
      const bool mine = leader && l < j0 + k;
      bool got = false;
      if (mine) {
        uint64_t old = atom_add_acq(&d.tag[line], PIN1);  // line data is read after the pin
        uint64_t ost = tag_state(old);
        got = tag_page(old) == pg && (ost == ST_READY || ost == ST_MODIFIED);
        if (!got) cache_unpin(d, line);  // evicted since the probe
      }
      __syncwarp();  // the pins' acquires come before every lane's reads of the lines
      const unsigned lost = __ballot_sync(kFull, mine && !got);
      uint32_t myline = __shfl_sync(kFull, line, lead_lane & 31);
      if (lost) {
        // rows of a lost page and those behind the first of them come in the next round
        unsigned gone = __ballot_sync(kFull, act && ((lost >> (lead_lane & 31)) & 1u)) >> j0;
        k = min(k, (uint32_t)(__ffs(gone) - 1));
      }
      if (k) sum_rows<MF4>(d, j0, k, myline, off, nf4, acc);
      __syncwarp();
      if (got) cache_unpin(d, line);
      j0 += k;
      if (k) continue;
    }
    // row j0's page is not READY: wait for it
    uint64_t pj = __shfl_sync(kFull, pg, j0 & 31);
    uint32_t lj;
    if (!warp_pin_page(d, pj, a.q0, a.deadline, lj)) return false;
    sum_rows<MF4>(d, j0, 1, lj, off, nf4, acc);
    __syncwarp();
    if (l == 0) cache_unpin(d, lj);
    j0 += 1;
  }
  return true;
}


// ================================================================ completion side
// Release what a completed command held (Sec. 3.2.1): the line becomes READY (or
// INVALID on an error), the share-table entry is removed, the transaction barrier
// (completion word) is set, the slot returns to EMPTY and the in-flight count drops.
// The caller's fence after it read the completion entry orders the device's data before
// the line's new state; one more fence orders everything before the slot and the
// in-flight entry are free again.
__device__ __forceinline__ void complete_command(const Dev &d, uint32_t q, uint32_t cid, uint32_t status) {
  uint64_t i = (uint64_t)q * d.depth + cid;
  uint64_t ctx = ld_rlx64(&d.cmd_ctx[i]);
  uint64_t st = ld_rlx64(&d.sqe_state[i]);
  uint64_t ticket = st >> 2;
  uint64_t kind = ctx >> 60;
  uint32_t sh = (uint32_t)(ctx >> 32) & 0x0FFFFFFFu;
  uint32_t idx = (uint32_t)ctx;
  if (kind == CTX_FILL) {
    if (status == 0) {
      atomicAdd(&d.tag[idx], 1ull);  // BUSY (1) -> READY (2)
    } else {
      atomicAnd(&d.tag[idx], PIN_MASK);  // back to INVALID
    }
  } else if (kind == CTX_WB) {
    if (idx) atomicAnd(&d.tag[idx - 1], ~TAG_WB);  // flush write-back from the line itself
  }
  const bool entry = kind == CTX_FILL || kind == CTX_WB || kind == CTX_BUF;
  if (entry) st_rlx64(&d.sh_val[sh], 0ull);
  if (status) atomicAdd(stat_ptr(d, S_IO_ERRORS), 1ull);
  st_rlx64(&d.cmpl[i], ((ticket & 0xFFFFFFFFull) << 32) | ((uint64_t)(status & 0x7FFF) << 1) | 1ull);
  fence_ar();
  if (entry) sh_clear(d, sh);
  st_rlx64(&d.sqe_state[i], (ticket << 2) | SQE_EMPTY);
  atomicAdd(&d.sq_resv[q], (unsigned long long)(-(int64_t)(1ull << 32)));
}

// Alg. 1, warp-centric CQ polling of queue q: lane l checks entry offset+l of the
// current 32-entry window against the expected phase; the mask accumulates found
// entries (they may arrive in any order); a full mask advances the head and rings the
// CQ doorbell.  The CQ has twice as many entries as the SQ, so with at most depth-1
// commands outstanding and at most 31 consumed entries in the open window it never
// fills (the device never has to wait for CQ space).
// A dedicated poller keeps its position in registers (PollPos) for the whole launch.
struct PollPos {
  uint32_t offset, mask, phase;
};
__device__ __forceinline__ PollPos poll_load(const Dev &d, uint32_t q) {
  const uint32_t *ps = &d.cq_poll[q * 4];
  return PollPos{ld_rlx32(&ps[0]), ld_rlx32(&ps[1]), ld_rlx32(&ps[2])};
}
__device__ __forceinline__ void poll_store(const Dev &d, uint32_t q, const PollPos &p) {
  uint32_t *ps = &d.cq_poll[q * 4];
  __syncwarp();
  if (lane_id() == 0) {
    st_rlx32(&ps[0], p.offset);
    st_rlx32(&ps[1], p.mask);
    st_rlx32(&ps[2], p.phase);
  }
  __syncwarp();
}
static __device__ bool cq_poll(const Dev &d, uint32_t q, PollPos &p) {
  unsigned l = lane_id();
  uint32_t found = 0, windows = 0;
  for (int win = 0; win < 4; ++win) {
    bool valid = false;
    uint32_t w3 = 0;
    if (!((p.mask >> l) & 1u)) {
      w3 = ld_rlx32(&d.cq[(uint64_t)q * d.cq_size + p.offset + l].dw[3]);
      valid = ((w3 >> 16) & 1u) == p.phase;
    }
    unsigned b = __ballot_sync(kFull, valid);
    if (!b) break;
    fence_ar();  // an entry's phase was read: what the device wrote before it is visible now
    if (valid) complete_command(d, q, w3 & 0xFFFFu, w3 >> 17);
    found += __popc(b);
    p.mask |= b;
    if (p.mask != kFull) break;
    p.mask = 0;
    p.offset += 32;
    if (p.offset >= d.cq_size) {
      p.offset = 0;
      p.phase ^= 1u;
    }
    ++windows;
    __syncwarp();
    if (l == 0) st_rel32(&d.cq_db[q], p.offset);
  }
  __syncwarp();
  if (l == 0) {
    if (found) atomicAdd(stat_ptr(d, S_CQES), (unsigned long long)found);
    if (windows) atomicAdd(stat_ptr(d, S_CQ_DOORBELLS), (unsigned long long)windows);
  }
  __syncwarp();
  return found != 0;
}

// ================================================================ emulated device
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The emulated NVMe device.  Every service warp is one of its engines and may serve
// any queue.  Per queue the device keeps (unwrapped counters): `fetch`, the next SQE to
// take; `seen`, how far the doorbell has been observed (commands below it carry their
// arrival time); `cqt`, the next CQ slot.  An engine takes up to kEmuBatch due commands
// in SQ order by compare-and-swap on `fetch` (a command is due once its latency has
// elapsed and the queue's throughput budget allows it), moves the pages between the
// store (pinned host memory, over the host link) and HBM, then reserves CQ slots and
// posts the CQEs {SQ head, SQ id, CID, status, phase}.  Commands of one queue complete
// in any order, as NVMe allows.
constexpr uint32_t kEmuBatch = 2;
constexpr uint64_t kEmuSlackNs = 16000;

// Returns the number of commands served, or kEmuDevFull when commands were due but
// their device was booked, or kEmuLost when another engine took them.  f, db: the queue's fetch counter and doorbell as the caller's
// scan has read them (uniform; db at least one command ahead).  block_dev: a device this
// call may not book (a demand command of the same engine pass is waiting for it), ~0u
// for none.
constexpr uint32_t kEmuDevFull = 0x80000000u, kEmuLost = 0x40000000u;
static __device__ uint32_t emu_serve(const Dev &d, uint32_t q, uint32_t f, uint32_t db, uint32_t block_dev = ~0u) {
  unsigned l = lane_id();
  uint32_t k = 0, full = 0;
  uint64_t now = gtimer();
  const uint32_t dv = d.ndev > 1 ? q % d.ndev : 0u;  // the device this queue belongs to
  const bool model = d.lat_ns || d.ns_per_page || d.ns_rd_dev || d.ns_wr_dev;
  fence_ar();  // the doorbell was read: the commands below it are visible now
  __syncwarp();
  int4 ea = make_int4(0, 0, 0, 0), eb = ea, ec = ea, eg = ea;
  auto read_entry = [&]() {
    if (l < k) {
      const uint32_t *e = d.sq[(uint64_t)q * d.depth + ((f + l) & d.dmask)].dw;
      ea = ld_cg16(e);
      eb = ld_cg16(e + 4);
      ec = ld_cg16(e + 8);
      eg = ld_cg16(e + 12);
    }
  };
  if (!model) {
    // no latency model: every command the doorbell exposes is due at once.  Both counters
    // only grow, so with f still current (checked by the compare-and-swap) the
    // commands [f, db) are unfetched whichever of the two was read first.  The entries
    // are read beside the compare-and-swap and used only if it succeeds.
    k = min(db - f, kEmuBatch);
    uint32_t got = f;
    if (l == 0) got = atomicCAS(&d.emu_fetch[q], f, f + k);
    read_entry();
    got = __shfl_sync(kFull, got, 0);
    if (got != f) return kEmuLost;
  } else if (l == 0) {
    uint32_t seen = ld_acq32(&d.emu_seen[q]);
    db = ld_acq32(&d.sq_db[q]);
    // stamp the arrival of commands the doorbell has newly exposed, then publish them
    uint32_t fresh = db - seen;
    if ((int32_t)fresh > 0) {
      for (uint32_t i = 0; i < fresh; ++i)
        st_rlx64(&d.emu_arrival[(uint64_t)q * d.depth + ((seen + i) & d.dmask)], now);
      fence_ar();
      atomicCAS(&d.emu_seen[q], seen, seen + fresh);
      seen = ld_acq32(&d.emu_seen[q]);
    }
    f = ld_rlx32(&d.emu_fetch[q]);
    uint32_t avail = seen - f;
    if ((int32_t)avail > 0) {
      if (avail > kEmuBatch) avail = kEmuBatch;
      while (k < avail) {
        uint64_t arr = ld_rlx64(&d.emu_arrival[(uint64_t)q * d.depth + ((f + k) & d.dmask)]);
        if (now < arr + d.lat_ns) break;
        ++k;
      }
      if (k && dv == block_dev) {
        k = 0;
        full = kEmuDevFull;
      }
      // Throughput: the batch is booked on the queue's pipe and on its device when each
      // is free (reads and writes take device time of their own).  Bookings follow each
      // other without gaps while the pipe has been idle for less than kEmuSlackNs
      // (engines poll in turns, so a pipe's next batch is picked up a little late): a
      // token bucket that may run kEmuSlackNs ahead after a pause, which moves the
      // long-run rate by less than kEmuSlackNs per pause.  Bookings of a batch that is
      // not served after all (another booking failed, or another engine took the
      // commands meanwhile) are given back.
      uint64_t qcost = d.ns_per_page * k, dcost = 0;
      bool qbooked = false, dbooked = false;
      if (k && qcost) {
        uint64_t busy = ld_rlx64(&d.emu_busy[q]);
        if (busy > now) {
          k = 0;
        } else {
          uint64_t nb = (busy + kEmuSlackNs > now ? busy : now) + qcost;
          qbooked = atomicCAS(&d.emu_busy[q], (unsigned long long)busy, (unsigned long long)nb) == busy;
          if (!qbooked) k = 0;
        }
      }
      if (k && (d.ns_rd_dev || d.ns_wr_dev)) {
        for (uint32_t i = 0; i < k; ++i) {
          uint32_t op = ld_rlx32(&d.sq[(uint64_t)q * d.depth + ((f + i) & d.dmask)].dw[0]) & 0xFFu;
          dcost += op == OP_WRITE ? d.ns_wr_dev : (op == OP_READ ? d.ns_rd_dev : 0);
        }
        uint64_t busy = ld_rlx64(&d.dev_busy[dv]);
        if (busy > now) {
          k = 0;
          full = kEmuDevFull;
        } else {
          uint64_t nb = (busy + kEmuSlackNs > now ? busy : now) + dcost;
          dbooked = atomicCAS(&d.dev_busy[dv], (unsigned long long)busy, (unsigned long long)nb) == busy;
          if (!dbooked) k = 0;
        }
      }
      if (k && atomicCAS(&d.emu_fetch[q], f, f + k) != f) k = 0;
      if (!k) {
        if (qbooked) atomicAdd(&d.emu_busy[q], (unsigned long long)(-(int64_t)qcost));
        if (dbooked && dcost) atomicAdd(&d.dev_busy[dv], (unsigned long long)(-(int64_t)dcost));
      }
    }
  }
  if (model) {
    k = __shfl_sync(kFull, k, 0);
    if (!k) return __shfl_sync(kFull, full, 0);
    f = __shfl_sync(kFull, f, 0);
    __syncwarp();  // lane 0's acquire of the doorbell orders the reads of every lane
    read_entry();
  }
  // the places of the completions, taken while the data moves (a completion queue holds
  // every command in flight twice over)
  uint32_t slot0 = 0;
  if (l == 0) slot0 = atomicAdd(&d.emu_cqt[q], k);
  // command fields: lane i < k holds those of SQE f+i
  uint32_t dw0 = 0, nlb = 0, status = 0;
  uint64_t prp1 = 0, slba = 0, t_commit = 0;
  bool drop = false;
  if (l < k) {
    const int4 a = ea, b = eb, c = ec, g = eg;
    dw0 = (uint32_t)a.x;
    t_commit = (uint64_t)(uint32_t)a.z | ((uint64_t)(uint32_t)a.w << 32);
    prp1 = (uint64_t)(uint32_t)b.z | ((uint64_t)(uint32_t)b.w << 32);
    slba = (uint64_t)(uint32_t)c.z | ((uint64_t)(uint32_t)c.w << 32);
    nlb = (uint32_t)g.x & 0xFFFFu;
    uint32_t opcode = dw0 & 0xFFu;
    uint64_t nbytes = ((uint64_t)nlb + 1) * 512;
    // from here on slba is the store page of the command (block on device dv)
    slba = (d.ndev > 1 ? (slba / (kPage / 512)) * d.ndev + dv : slba / (kPage / 512));
    if (opcode != OP_FLUSH && (slba * kPage + nbytes > d.store_bytes || nbytes != kPage)) status = 0x80;
    if (d.fault_flags) {
      uint64_t h = mix64(d.seed ^ ((uint64_t)q << 40) ^ (uint64_t)(f + l));
      if ((uint32_t)(h >> 32) < d.fault_thresh) {
        if (d.fault_flags & 1u) status = 0x6;
        if (d.fault_flags & 2u) drop = true;
      }
    }
  }
  // data movement: every page of the batch has its loads in flight before any store
  int4 v[kEmuBatch][8];
  uint64_t srcs[kEmuBatch], dsts[kEmuBatch];
  bool mv[kEmuBatch];
#pragma unroll
  for (uint32_t j = 0; j < kEmuBatch; ++j) {
    uint32_t opj = __shfl_sync(kFull, dw0, j) & 0xFFu;
    uint32_t stj = __shfl_sync(kFull, status, j);
    uint64_t pj = __shfl_sync(kFull, prp1, j), sj = __shfl_sync(kFull, slba, j);
    mv[j] = j < k && stj == 0 && (opj == OP_READ || opj == OP_WRITE);
    srcs[j] = opj == OP_READ ? (uint64_t)(d.store + sj * kPage) : pj;
    dsts[j] = opj == OP_READ ? pj : (uint64_t)(d.store + sj * kPage);
    if (mv[j]) {
      const int4 *sp = (const int4 *)srcs[j];
#pragma unroll
      for (int t = 0; t < 8; ++t) v[j][t] = ld_cg16(sp + t * 32 + l);
    }
  }
  uint32_t rd = 0, wr = 0;
#pragma unroll
  for (uint32_t j = 0; j < kEmuBatch; ++j) {
    if (mv[j]) {
      int4 *dp = (int4 *)dsts[j];
#pragma unroll
      for (int t = 0; t < 8; ++t) st_cg16(dp + t * 32 + l, v[j][t]);
      if ((__shfl_sync(kFull, dw0, j) & 0xFFu) == OP_READ) ++rd;
      else ++wr;
    }
  }
  // per-page accounting of the data moved (lane i counts command i)
  if (l < k && status == 0) {
    uint32_t opcode = dw0 & 0xFFu;
    if (opcode == OP_READ) atomicAdd(&d.pg_reads[slba], 1u);
    else if (opcode == OP_WRITE) atomicAdd(&d.pg_writes[slba], 1u);
  }
  __syncwarp();
  // completion entries: the release of each orders the whole warp's data before it
  slot0 = __shfl_sync(kFull, slot0, 0);
  if (l < k) {
    uint32_t sl = slot0 + l;
    uint32_t pos = sl % d.cq_size;
    uint32_t phase = ((sl / d.cq_size) & 1u) ^ 1u;
    Cqe *c = &d.cq[(uint64_t)q * d.cq_size + pos];
    uint32_t cid = dw0 >> 16;
    if (d.trace) {
      uint32_t ti = atomicAdd(d.trace_n, 1u);
      if (ti < d.trace_cap) {
        TraceRec *tr = &d.trace[ti];
        tr->page = slba;
        tr->t_seen = model
                         ? ld_rlx64(&d.emu_arrival[(uint64_t)q * d.depth + ((f + l) & d.dmask)])
                         : 0ull;
        tr->t_start = now;
        tr->t_done = gtimer();
        tr->q = q;
        tr->cid = cid;
        tr->opcode = dw0 & 0xFFu;
        tr->status = status | (drop ? 0x10000u : 0u);
        tr->t_commit = t_commit;
      }
    }
    if (drop) {
      // the completion is lost; leave a harmless entry with the old phase
      st_rlx32(&c->dw[2], (q << 16) | ((f + l + 1) & d.dmask));
    } else {
      st_rlx32(&c->dw[0], 0u);
      st_rlx32(&c->dw[1], 0u);
      st_rlx32(&c->dw[2], (q << 16) | ((f + l + 1) & d.dmask));
      st_rel32(&c->dw[3], cid | (phase << 16) | (status << 17));
    }
  }
  if (l == 0) {
    atomicAdd(stat_ptr(d, S_COMMANDS), (unsigned long long)k);
    if (rd) atomicAdd(stat_ptr(d, S_BYTES_READ), (unsigned long long)rd * kPage);
    if (wr) atomicAdd(stat_ptr(d, S_BYTES_WRITTEN), (unsigned long long)wr * kPage);
  }
  __syncwarp();
  return k;
}

// ================================================================ engine
// One cooperative launch per library call, one CTA per SM.  Of 19 CTAs three (evenly spread)
// are service CTAs: their warps poll the completion queues (Alg. 1), one queue each where
// there are enough of them, and are the engines of the emulated device for every queue.
// The warps of the others run the application.  Service on SMs of its own, because the
// miss path is bound by instruction supply as much as by L2 round trips: next to the
// service loops a warp met 260 instruction-cache misses in a round of misses (ncu: 18 %
// of an SM's fetches), and a computing warp slows the device down.
// A launch of few CTAs has a service warp in each CTA instead, which does both.
// No kernel of the library ever waits on another launch: the device, the pollers and the
// waiters are co-resident warps of one grid, and every wait is bounded by a deadline.
constexpr uint32_t kServiceNum = 3, kServiceDen = 19;  // 24 of 152 CTAs: 2,048 application warps are left
struct Roles {
  uint32_t svc;       // service CTAs (0: a service warp in every CTA)
  uint32_t app_ctas;  // CTAs with application warps
  uint32_t per_cta;   // application warps of each of them
};
__host__ __device__ __forceinline__ Roles engine_roles(uint32_t grid, uint32_t warps) {
  Roles r;
  r.svc = grid >= 8 ? grid * kServiceNum / kServiceDen : 0;
  r.app_ctas = grid - r.svc;
  r.per_cta = r.svc ? warps : warps - 1;
  return r;
}
// `sw`: this engine's number (rotation start); the first `pollers` engines poll when `poll`.
static __device__ void service_loop(const Dev &d, uint32_t app_ctas, uint64_t deadline, bool poll, uint32_t sw,
                                    uint32_t pollers) {
  unsigned l = lane_id();
  uint32_t ns = 32, empty = 0;
  for (uint32_t iter = 0;; ++iter) {
    bool progress = false, lost = false;
    // device engine: serve one queue per iteration, one with work from a window of 32
    // queues: its home queue first, which with every queue busy leaves few engines after
    // the same commands, else one that rotates and differs between engines
    // (the doorbells and fetch counters of a window are two 128-byte lines read in one
    // round trip; they only select a queue, emu_serve checks them again.  Reading all
    // 128 queues in every pass of every engine kept those few lines so busy that the
    // threads' own doorbells and the compare-and-swaps on them queued up behind)
    // (demand queues first: the prefetch queues are served only when no demand queue
    // has a command the device may take now; a prefetch queue does not book a device
    // that a due demand command found booked in this pass, so the device's next free
    // turn goes to the demand command)
    uint32_t block_dev = ~0u;
#pragma unroll 1
    for (uint32_t cls = 0; cls < 2 && !progress; ++cls) {
      const uint32_t base = cls ? d.Q - d.Qp : 0u, cnt = cls ? d.Qp : d.Q - d.Qp;
      if (cnt == 0) continue;
      const uint32_t windows = (cnt + 31) / 32;
      // without prefetch queues any window will do; with them every demand queue is
      // looked at before the first prefetch queue
      const uint32_t looks = d.Qp ? windows : 1u;
      // its home queue's window unless that was empty last time; every fourth look goes
      // round all of them (more queues than engines)
      const uint32_t home = sw % cnt;
      const bool stray = (iter & 3) == 3;
      uint32_t w = windows == 1 ? 0u : (stray ? (iter >> 2) + sw : (home >> 5) + empty) % windows;
      uint32_t qsel = ~0u, f = 0, db = 0;
      for (uint32_t k = 0; k < looks && qsel == ~0u; ++k) {
        const uint32_t off = w * 32 + l;
        uint32_t dbv = 0, fv = 0;
        if (off < cnt) {
          dbv = ld_rlx32(&d.sq_db[base + off]);
          fv = ld_rlx32(&d.emu_fetch[base + off]);
        }
        unsigned m = __ballot_sync(kFull, (int32_t)(dbv - fv) > 0);
        if (m) {
          const uint32_t turn = ((sw * 31 + iter) * 0x9E3779B1u) >> 27;  // engines start at different queues
          int at = (__ffs(__funnelshift_r(m, m, turn)) - 1 + turn) & 31;
          if (!stray && w == home >> 5 && (m >> (home & 31)) & 1u) at = home & 31;
          qsel = base + w * 32 + at;
          f = __shfl_sync(kFull, fv, at);
          db = __shfl_sync(kFull, dbv, at);
        }
        if (++w == windows) w = 0;
      }
      if (qsel == ~0u) ++empty;
      else empty = 0;
      if (qsel != ~0u) {
        uint32_t r = emu_serve(d, qsel, f, db, block_dev);
        if (r == kEmuDevFull) block_dev = d.ndev > 1 ? qsel % d.ndev : 0u;
        else if (r == kEmuLost) lost = true;
        else if (r) progress = true;
      }
    }
    // completion side (Alg. 1) for the queues this warp polls
    if (poll)
      for (uint32_t q = sw; q < d.Q; q += pollers) {
        PollPos p = poll_load(d, q);
        if (cq_poll(d, q, p)) {
          poll_store(d, q, p);
          progress = true;
        }
      }
    if (progress || (lost && (iter & 7) != 7)) {  // another engine was faster: there is work, look again at once
      ns = 32;
      continue;
    }
    uint32_t done = 0;
    if (l == 0) done = ld_acq32(&d.run->app_done);
    done = __shfl_sync(kFull, done, 0);
    if (done >= app_ctas) {
      bool drained = true;
      for (uint32_t q = l; q < d.Q; q += 32)
        if ((ld_acq64(&d.sq_resv[q]) >> 32) != 0) drained = false;
      if (__all_sync(kFull, drained)) break;
    }
    if (gtimer() > deadline) {
      if (l == 0) set_error(d, -110);
      break;
    }
    __nanosleep(ns);
    ns = ns < 256 ? ns * 2 : 256;
  }
}

// A dedicated Alg. 1 poller of the queues q, q + step, ...  Ends when every application
// warp is done and its queues have nothing in flight.
static __device__ void poller_loop(const Dev &d, uint32_t q0, uint32_t step, uint32_t app_ctas, uint64_t deadline) {
  unsigned l = lane_id();
  const bool one = q0 + step >= d.Q;
  PollPos p = poll_load(d, q0);
  for (uint32_t iter = 1;; ++iter) {
    bool found = false;
    if (one) {
      found = cq_poll(d, q0, p);
    } else {
      for (uint32_t q = q0; q < d.Q; q += step) {
        p = poll_load(d, q);
        if (cq_poll(d, q, p)) {
          poll_store(d, q, p);
          found = true;
        }
      }
    }
    if (found) continue;
    if (iter & 3) {  // the end of the call is looked for now and then
      __nanosleep(32);
      continue;
    }
    uint32_t done = 0;
    if (l == 0) done = ld_acq32(&d.run->app_done);
    done = __shfl_sync(kFull, done, 0);
    if (done >= app_ctas) {
      bool drained = true;
      for (uint64_t q = q0 + (uint64_t)l * step; q < d.Q; q += 32ull * step)
        if ((ld_acq64(&d.sq_resv[q]) >> 32) != 0) drained = false;
      if (__all_sync(kFull, drained)) break;
    }
    if (gtimer() > deadline) {
      if (l == 0) set_error(d, -110);
      break;
    }
  }
  if (one) poll_store(d, q0, p);
}

// Grid barrier over the application warps only (service warps never join).  The warps of a
// CTA meet in shared memory; the last one of each meets the others' in device memory (a
// single counter for all 2,000 warps took 5 us of serialised atomics).
static __device__ bool app_barrier(const Dev &d, uint64_t deadline) {
  CtaState &cs = cta_state();
  bool ok = true;
  __syncwarp();
  if (lane_id() == 0) {
    volatile uint32_t *cgen = &cs.bar_gen;
    const uint32_t mine = *cgen;
    fence_ar();
    if (atomicAdd(&cs.bar_count, 1u) + 1 == cs.active) {
      cs.bar_count = 0;
      fence_ar();
      uint32_t gen = ld_acq32(&d.run->bar_gen);
      if (atomicAdd(&d.run->bar_count, 1u) + 1 == cs.ctas_active) {
        st_rlx32(&d.run->bar_count, 0u);
        fence_ar();
        st_rel32(&d.run->bar_gen, gen + 1);
      } else {
        uint32_t spin = 0;
        while (ld_acq32(&d.run->bar_gen) == gen) {
          if ((++spin & 15) == 0 && gtimer() > deadline) {
            set_error(d, -110);
            ok = false;
            break;
          }
          __nanosleep(64);
        }
      }
      fence_ar();
      if (ok) *cgen = mine + 1;
    } else {
      uint32_t spin = 0;
      while (*cgen == mine) {
        if ((++spin & 15) == 0 && gtimer() > deadline) {
          set_error(d, -110);
          ok = false;
          break;
        }
        __nanosleep(64);
      }
      fence_ar();
    }
  }
  ok = __shfl_sync(kFull, ok, 0);
  __syncwarp();
  return ok;
}


// Slice queue of long rows (BFS: one per level parity, SpMV: 0).  own_work_done: this warp
// queues no more slices (counted per CTA; lane 0).  slices_end: whether the queue is known to end at or before
// ticket k (lane 0; `phase`: the level).  One warp of a CTA watches the shared counters for
// the others, which look at shared memory: 2,000 warps polling one line would keep it from
// the warps that still work, and polling seldom costs every level several microseconds.
static __device__ __forceinline__ void own_work_done(const Dev &d, uint32_t par) {
  CtaState &cs = cta_state();
  fence_ar();
  if (atomicAdd(&cs.own_done, 1u) + 1 == cs.active) {
    cs.own_done = 0;
    fence_ar();
    atomicAdd(&d.run->units_done[par], 1u);
  }
}
static __device__ __forceinline__ bool slices_end(const Dev &d, uint32_t par, uint32_t phase, uint32_t k) {
  CtaState &cs = cta_state();
  volatile uint32_t *seen = &cs.end_seen, *count = &cs.end_count;
  if (*seen != phase + 1 && atomicCAS(&cs.watched, 0u, 1u) == 0u) {
    if (ld_acq32(&d.run->units_done[par]) >= cs.ctas_active) {
      *count = ld_acq32(&d.run->hub_count[par]);
      __threadfence_block();
      *seen = phase + 1;
    }
    atomicExch(&cs.watched, 0u);
  }
  if (*seen != phase + 1) return false;
  __threadfence_block();
  return *count <= k;
}

// Occupancy the engine is compiled for, in groups of kWarps warps per SM (register
// budget): App::kMinBlocks if the application asks for more, else 2
template <class App, class = void>
struct MinBlocks {
  static constexpr int value = 2;
};
template <class App>
struct MinBlocks<App, decltype((void)App::kMinBlocks, void())> {
  static constexpr int value = App::kMinBlocks;
};
// CTAs that share an SM: one, which has all of its warps, unless the application asks for more
template <class App, class = void>
struct CtasPerSm {
  static constexpr int value = 1;
};
template <class App>
struct CtasPerSm<App, decltype((void)App::kCtasPerSm, void())> {
  static constexpr int value = App::kCtasPerSm;
};
template <class App>
struct EngineShape {
  static constexpr int ctas = CtasPerSm<App>::value;
  static constexpr int warps = kWarps * MinBlocks<App>::value / ctas;
  static constexpr int threads = warps * 32;
};
// A user's application: its CTAs have kWarps warps, so that what it keeps for each warp of
// a CTA is sized by kWarps.  Of its members only run() and kMinBlocks mean anything here.
template <class App>
struct UserApp {
  static constexpr int kMinBlocks = MinBlocks<App>::value, kCtasPerSm = kMinBlocks;
  App app;
  __device__ __forceinline__ void run(const Dev &d, const AppCtx &a) const { app.run(d, a); }
};
// dynamic shared memory an application wants for each warp of the CTA
template <class App, class = void>
struct SharedPerWarp {
  static constexpr int value = 0;
};
template <class App>
struct SharedPerWarp<App, decltype((void)App::kSharedPerWarp, void())> {
  static constexpr int value = App::kSharedPerWarp;
};
template <class App>
constexpr int engine_shared() {
  return SharedPerWarp<App>::value * EngineShape<App>::warps;
}

// An application with nothing to do says so with
//   __device__ bool idle(const Dev &d) const;
// (the same answer in every thread of the launch): its engine ends at once.
template <class App, class = void>
struct HasIdle {
  static constexpr bool value = false;
};
template <class App>
struct HasIdle<App, decltype((void)&App::idle)> {
  static constexpr bool value = true;
};

template <class App>
__global__ void __launch_bounds__(EngineShape<App>::threads, EngineShape<App>::ctas)
    engine_kernel(const __grid_constant__ Dev d, const __grid_constant__ App app) {
  if constexpr (HasIdle<App>::value) {
    if (app.idle(d)) return;
  }
  constexpr uint32_t kCtaWarps = EngineShape<App>::warps;
  const Roles r = engine_roles(gridDim.x, kCtaWarps);
  // service CTAs are evenly spread over the grid
  const uint32_t before = (uint32_t)((uint64_t)blockIdx.x * r.svc / gridDim.x);
  const bool svc_cta = (uint32_t)(((uint64_t)blockIdx.x + 1) * r.svc / gridDim.x) != before;
  const uint32_t app_cta = blockIdx.x - before;
  const uint32_t n_app = r.app_ctas * r.per_cta;
  const uint32_t n_active = (d.app_active && d.app_active < n_app) ? d.app_active : n_app;
  CtaState &cs = cta_state();
  static_assert(sizeof(Dev) % 4 == 0, "copied in 4-byte words");
  for (uint32_t i = threadIdx.x; i < sizeof(Dev) / 4; i += EngineShape<App>::threads)
    ((uint32_t *)&cs.dev)[i] = ((const uint32_t *)&d)[i];
  if (threadIdx.x == 0) {
    cs.done = cs.bar_count = cs.bar_gen = cs.own_done = cs.watched = cs.end_seen = cs.end_count = 0;
    cs.active = n_active > app_cta ? (n_active - app_cta + r.app_ctas - 1) / r.app_ctas : 0;
    cs.ctas_active = n_active < r.app_ctas ? n_active : r.app_ctas;
  }
  __syncthreads();
  uint32_t warp = threadIdx.x >> 5;
  uint64_t deadline = gtimer() + (d.session_ns ? d.session_ns : d.timeout_ns);
  AppCtx a;
  // consecutive application warps are on different CTAs: a call that runs a few hundred
  // warps has them on as many SMs, and they seldom wait for each other's issue slots
  const uint32_t first_app = kCtaWarps - r.per_cta;
  a.warp = (warp - first_app) * r.app_ctas + app_cta;
  a.n_warps = n_active;
  bool serve = true, poll = false;
  uint32_t sw = blockIdx.x;
  if (svc_cta) {
    const uint32_t n_svc = r.svc * kCtaWarps, me = warp * r.svc + before;
    const uint32_t n_poll = min(d.Q, n_svc / 3);
    if (me < n_poll) {
      poller_loop(d, me, n_poll, r.app_ctas, deadline + d.timeout_ns);
      return;
    }
    sw = me - n_poll;
  } else if (warp < first_app) {
    poll = true;
  } else {
    // application warps beyond n_active are not needed by this call (the working set of the
    // active ones stays in the cache)
    if (a.warp < n_active) {
      // home queue by thread index, spread so that the lanes of a warp and the lane 0 of
      // consecutive warps all start on different queues
      a.q0 = (uint32_t)((a.warp + (uint64_t)lane_id() * ((d.Q + 31) / 32)) % d.Q);
      a.deadline = deadline;
      app.run(d, a);
      __syncwarp();
    }
    if (lane_id() == 0) {
      fence_ar();
      if (atomicAdd(&cs.done, 1u) + 1 == r.per_cta) {
        fence_ar();
        atomicAdd(&d.run->app_done, 1u);
      }
    }
    serve = a.warp >= n_active && a.warp - n_active < d.extra_engines;
    sw = gridDim.x + a.warp;
  }
  // (one call site: the engines of an SM share its instruction cache)
  if (serve) service_loop(d, r.app_ctas, deadline + d.timeout_ns, poll, sw, gridDim.x);
}

}  // namespace agile
