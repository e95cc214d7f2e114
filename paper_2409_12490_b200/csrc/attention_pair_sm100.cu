// K4 / K5 for 16-bit heads of 128 channels, by pairs of CTAs that share their tensor cores' operands (tcgen05 cta_group::2): the kernel
// for launches of few or short units.  Same results as attention_sm100.cu, bit for bit: the same products in the same order.
//
// There a unit of 256 query rows occupies one SM, with one S buffer per query tile: S -> softmax -> P -> P V -> next S is a serial
// chain.  Here two SMs share a unit: every MMA is M = 256, each CTA holds its own 128 rows of Q, S, P and O and half of every K tile (64
// keys) and V tile (64 channels), so that a K/V tile pair still costs an SM 32 KB per 128 x 128 logits, and with one query tile per
// CTA tensor memory has room for three S tiles.  A unit takes about half as long, and its first tiles run under the end of the one
// before.  Roles of a CTA (512 threads):
//   warps 0-3, 4-7  softmax, one thread per query row; the two warpgroups take the K/V tiles in turn
//   warps 8-11      epilogue: O / l -> shared memory -> global (TMA stores)
//   warp  12        TMA producer of Q and K       warp 13  TMA producer of V
//   warp  14        MMA issuer of the pair (first CTA only)
//   warp  15        scheduler
// Tensor memory (512 columns): S_0 | S_1 | S_2 | O, 128 fp32 columns each; P goes over the first half of its S.
// QK^T runs three tiles ahead of P V, across the ends of units.  The reference maximum of a row goes from tile to tile, from one warpgroup
// to the other; what each tile adds to the row's sum goes to the epilogue warps, which add up in the tiles' order.  O is rescaled (only when
// the maximum grew by more than 2^8) by the threads that form the tile's P.
// What bounds a unit: a tile's P -> P V -> QK^T three tiles on -> softmax (1800 + 2900 cycles) over three S buffers, 1600 to 1850 cycles per
// tile against 1040 of MMAs; in long loops the power cap, where the other kernel takes less energy over long units.  Both kernels
// in graph replays, us (attention_sm100.cu / this one): 32 query / 8 KV heads, segment 512, block 32, budget 1024: 1300 tokens
// 32.3 / 29.1, 2000 38.0 / 33.8, 13000 187 / 177; 8 / 2 heads, segment 256, budget 2048: 1000 tokens 21.9 / 15.3, 2000 35.5 / 23.0;
// dense, 8 / 2 heads: 2000 tokens 35.0 / 22.4, 6000 108 / 79.  The line between them: pairs_are_faster in attention_sm100.cu.
#include "attention_units.cuh"

namespace cp {
namespace {

constexpr int kThreads = 512;
constexpr int kSlotBytes = 64 * 128 * 2;       // half a K tile (64 keys) or half a V tile (64 channels)
constexpr int kSlots = 3;                      // of K, V and S: tile g uses slot g % 3 of each
constexpr int kQBytes = 2 * kHalfBytes;        // 128 rows of Q
constexpr int kSmemQ = 0;                      // two units
constexpr int kSmemK = kSmemQ + 2 * kQBytes;
constexpr int kSmemV = kSmemK + kSlots * kSlotBytes;
constexpr int kSmemO = kSmemV + kSlots * kSlotBytes;     // 128 rows of O on their way out
constexpr int kSmemStat = kSmemO + kQBytes;
constexpr int kSched = 4;                      // published units: the MMA warp is up to three ahead of the epilogue
constexpr int kSums = 8;                        // tiles whose row sums wait to be added up
constexpr int kSmemSum = kSmemStat + kSched * kTile * 4;
constexpr int kSmemBar = kSmemSum + kSums * kTile * 8;
constexpr int kBarBytes = 4096;
constexpr int kSmemTotal = kSmemBar + kBarBytes + 1024;   // + slack to align the tiles to 1024 bytes

struct Bars {
  unsigned long long q_full[2], q_empty[2];
  unsigned long long k_full[kSlots], v_full[kSlots];
  unsigned long long s_full[kSlots];     // QK^T of a tile is complete: S may be read, and its K slot filled again
  unsigned long long p_full[kSlots];
  unsigned long long v_empty[kSlots];    // P V of a tile is complete: its V slot may be filled again, and O read
  unsigned long long o_full, o_empty;
  unsigned long long sum_full[kSums][4]; // per softmax warp: the row sums of its tile are there
  volatile uint32_t added[4];            // tiles whose row sums the epilogue warp has added up
  unsigned long long sched_full[kSched], sched_empty[kSched];
  unsigned long long clc_full;
  unsigned long long taken;              // both producers have begun the unit published last: the next one may be drawn
  __align__(16) uint32_t clc_resp[4];    // the hardware's answer to the last request for a further unit
  unsigned long long ref[2][kTile];      // a row's reference maximum after a tile of either warpgroup, and (upper half) that tile's number + 1
  int sched_unit[kSched];
  Unit sched_u[kSched];
  uint32_t mma_unit[4];                  // units between the MMA warp's QK^T and its P V: tiles | 2^31 if only the second CTA's rows see the last
  uint32_t tmem_base;
  volatile int abort_flag;
};
static_assert(sizeof(Bars) <= kBarBytes, "barrier block too small");

// Of q_full, k_full, v_full, p_full, o_empty and taken the first CTA's are used, for both CTAs: its MMA warp and scheduler wait on them.
// The MMA warp's commits arrive in both CTAs: q_empty, v_empty, s_full, o_full.
__device__ __forceinline__ uint32_t first_cta(const void* p) {      // the address of the first CTA's copy
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}
// An arrival at a barrier of the first CTA.  What it announces lies in tensor memory (complete by then: tcgen05.wait) or in nothing at
// all, so it needs no release at cluster scope, which waits for every outstanding store of the thread (more than 1000 cycles per tile).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Never suspends.  Like every test of a parity it is true before the phase that it asks about has begun, while the one before is open, so the
// caller has to know that that one is over.  v_full, ahead of a tile: the tile three before has gone through P V.  k_full, three tiles ahead of
// the next one: only if QK^T of that next tile has been issued, which it has not been (gq == gp + 1) where a unit ended and its successor was
// published too late; the wait then comes before the QK^T itself.  The other waits: each barrier's phases are waited for one after
// another by the same warp; s_full of every second tile by either softmax warpgroup, which has the tile before from the other one (row_get)
// by then; v_empty before a rescale: commits of one thread, in order, and s_full of a later one has been seen.
__device__ __forceinline__ bool mbar_ready(unsigned long long* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return __any_sync(0xffffffffu, ok != 0);
}
// Waits, and what is done once per unit, are kept out of the way of the instructions that every tile runs through: a branch over them
// costs the MMA warp some 80 cycles of instruction fetch.
#define CP_LIKELY(x) __builtin_expect(!!(x), 1)
#define CP_UNLIKELY(x) __builtin_expect(!!(x), 0)
__device__ __noinline__ bool wait_slow(unsigned long long* bar, uint32_t parity, Bars* bars, DeviceStatus* st, int site) {
  return mbar_wait(bar, parity, &bars->abort_flag, st, site);
}
__device__ __forceinline__ bool wait(unsigned long long* bar, uint32_t parity, Bars* bars, DeviceStatus* st, int site) {
  if (CP_LIKELY(mbar_test(bar, parity))) return true;
  return wait_slow(bar, parity, bars, st, site);
}
// A row's reference maximum after tile `tag` - 1, from the thread of the other warpgroup that has the same row.  Value and tag are one
// 8-byte word, written and read as one scalar (the parts of a vector access may be seen one without the other): a barrier would cost each side
// a hundred cycles and more per tile.  Every tile takes the value of the one before, also where it has no use for it (a unit's first),
// so neither side writes over a value that the other has not seen.
__device__ __forceinline__ void row_put(unsigned long long* p, float m, uint32_t tag) {
  asm volatile("{\n.reg .b64 v;\nmov.b64 v, {%1, %2};\nst.volatile.shared.b64 [%0], v;\n}" ::"r"(smem_u32(p)), "r"(__float_as_uint(m)), "r"(tag) : "memory");
}
__device__ __forceinline__ uint2 row_load(const unsigned long long* p) {
  uint2 v;
  asm volatile("{\n.reg .b64 v;\nld.volatile.shared.b64 v, [%2];\nmov.b64 {%0, %1}, v;\n}" : "=r"(v.x), "=r"(v.y) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __noinline__ bool row_wait(const unsigned long long* p, uint32_t tag, float* m, Bars* bars, DeviceStatus* st, int site) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    const uint2 v = row_load(p);
    *m = __uint_as_float(v.x);
    if (__all_sync(0xffffffffu, v.y == tag)) return true;
    if ((it & 255u) == 255u) {
      if (bars->abort_flag) return false;
      const unsigned long long now = globaltimer();
      if (t0 == 0) t0 = now;
      if (now - t0 > kWaitLimitNs) {
        bars->abort_flag = 1;
        report(st, CP_ERR_TIMEOUT, site, blockIdx.x, threadIdx.x, int(tag));
        return false;
      }
    }
  }
}
// `early`: what an earlier row_load found there, most often the value already
__device__ __forceinline__ bool row_get(const unsigned long long* p, uint2 early, uint32_t tag, float* m, Bars* bars, DeviceStatus* st, int site) {
  *m = __uint_as_float(early.x);
  if (CP_LIKELY(__all_sync(0xffffffffu, early.y == tag))) return true;
  float v;
  const bool ok = row_wait(p, tag, &v, bars, st, site);
  *m = v;
  return ok;
}
// until the epilogue warp has added up `tiles` tiles
__device__ __noinline__ bool wait_added(Bars* bars, int warp, uint32_t tiles, DeviceStatus* st) {
  const unsigned long long t0 = globaltimer();
  for (uint32_t it = 1; int32_t(bars->added[warp] - tiles) < 0; ++it) {
    if ((it & 255u) == 0) {
      if (bars->abort_flag) return false;
      if (globaltimer() - t0 > kWaitLimitNs) {
        bars->abort_flag = 1;
        report(st, CP_ERR_TIMEOUT, 16, blockIdx.x, threadIdx.x, int(tiles));
        return false;
      }
    }
  }
  return true;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// accumulates into the second CTA's rows only
__device__ __forceinline__ void umma2_ts_second(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p, e;\n.reg .b32 lid;\nelect.sync lid|e, 0xffffffff;\nsetp.eq.b32 p, 0, 0;\n"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, {%4, %4, %4, %4, %5, %5, %5, %5}, p;\n}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(0xffffffffu), "r"(0u) : "memory");
}
// eight MMAs (K = 128) by one elected lane, in one block: the descriptors advance by constants
__device__ __forceinline__ void umma2_qk8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile("{\n.reg .pred p, e;\n.reg .b32 lid;\n.reg .b64 a1,a2,a3,a4,a5,a6,a7,b1,b2,b3,b4,b5,b6,b7;\nelect.sync lid|e, 0xffffffff;\nsetp.ne.b32 p, 0, 0;\n"
    "add.s64 a1, %1, 2;\nadd.s64 a2, %1, 4;\nadd.s64 a3, %1, 6;\nadd.s64 a4, %1, 1024;\nadd.s64 a5, %1, 1026;\nadd.s64 a6, %1, 1028;\nadd.s64 a7, %1, 1030;\n"
    "add.s64 b1, %2, 2;\nadd.s64 b2, %2, 4;\nadd.s64 b3, %2, 6;\nadd.s64 b4, %2, 512;\nadd.s64 b5, %2, 514;\nadd.s64 b6, %2, 516;\nadd.s64 b7, %2, 518;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\nsetp.eq.b32 p, 0, 0;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], a4, b4, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a5, b5, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], a6, b6, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a7, b7, %3, p;\n}" ::"r"(d), "l"(a), "l"(b), "r"(idesc) : "memory");
}
__device__ __forceinline__ void umma2_pv8(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n.reg .pred p, e;\n.reg .b32 lid;\n.reg .b32 a1,a2,a3,a4,a5,a6,a7;\n.reg .b64 b1,b2,b3,b4,b5,b6,b7;\nelect.sync lid|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
    "add.s32 a1, %1, 8;\nadd.s32 a2, %1, 16;\nadd.s32 a3, %1, 24;\nadd.s32 a4, %1, 32;\nadd.s32 a5, %1, 40;\nadd.s32 a6, %1, 48;\nadd.s32 a7, %1, 56;\n"
    "add.s64 b1, %2, 128;\nadd.s64 b2, %2, 256;\nadd.s64 b3, %2, 384;\nadd.s64 b4, %2, 512;\nadd.s64 b5, %2, 640;\nadd.s64 b6, %2, 768;\nadd.s64 b7, %2, 896;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\nsetp.eq.b32 p, 0, 0;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a1], b1, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a2], b2, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a3], b3, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a4], b4, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a5], b5, %3, p;\n@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a6], b6, %3, p;\n"
    "@e tcgen05.mma.cta_group::2.kind::f16 [%0], [a7], b7, %3, p;\n}" ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void umma2_commit(unsigned long long* bar) {     // arrives in both CTAs
  asm volatile(
      "{\n.reg .pred e;\n.reg .b32 lid;\nelect.sync lid|e, 0xffffffff;\n"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}"
      ::"r"(smem_u32(bar)), "h"(uint16_t(3)) : "memory");
}
template <bool kF16> struct Idesc2 {          // M = 256
  static constexpr uint32_t qk = (Idesc<kF16>::qk & ~(0x1Fu << 24)) | ((256u >> 4) << 24);
  static constexpr uint32_t pv = (Idesc<kF16>::pv & ~(0x1Fu << 24)) | ((256u >> 4) << 24);
};

// ---------------------------------------------------------------- scheduler
// As in attention_sm100.cu, for the pair: the first CTA's scheduler requests, the answer arrives in both CTAs, and each CTA's
// scheduler decodes the unit and publishes it to its own warps.
template <int NS>
__device__ __forceinline__ void scheduler_role(const Args<NS>& a, Bars* bars, int rank, int lane) {
  for (uint32_t q = 0;; ++q) {
    const uint32_t slot = q % kSched;
    if (q >= kSched && !wait(&bars->sched_empty[slot], (q / kSched - 1) & 1, bars, a.st, 50)) return;
    int x = int(blockIdx.x >> 1);
    if (q > 0) {
      if (lane == 0) mbar_expect_tx(&bars->clc_full, 16);
      if (rank == 0) {
        if (!wait(&bars->taken, (q - 1) & 1, bars, a.st, 53)) return;
        __syncwarp();
        if (lane == 0)
          asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.multicast::cluster::all.b128 [%0], [%1];"
                       ::"r"(smem_u32(bars->clc_resp)), "r"(smem_u32(&bars->clc_full)) : "memory");
      }
      if (!wait(&bars->clc_full, (q - 1) & 1, bars, a.st, 52)) return;
      uint32_t ok, cta;
      asm volatile(
          "{\n.reg .pred p;\n.reg .b128 r;\nld.shared.b128 r, [%2];\n"
          "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\nselp.u32 %0, 1, 0, p;\nmov.u32 %1, 0;\n"
          "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, _, _, _}, r;\n}"
          : "=r"(ok), "=r"(cta) : "r"(smem_u32(bars->clc_resp)) : "memory");
      x = ok ? int(cta >> 1) : a.n_units;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the answer has been read before the next one is written
    }
    Unit u;
    if (x < a.n_units) u = prepare_unit(a, x, lane);
    if (lane == 0) {
      bars->sched_unit[slot] = x;
      if (x < a.n_units) bars->sched_u[slot] = u;
      mbar_arrive(&bars->sched_full[slot]);
    }
    if (x >= a.n_units) return;
    if (stop_requested(a, bars)) { bars->abort_flag = 1; return; }   // only this warp reads the status word in global memory
  }
}
constexpr uint32_t kReaders = 15;      // warps that receive every unit: 8 softmax, 4 epilogue, K and V producer, MMA
// The next unit with tiles, or of zeros; false at the end.  `taken`: see there (0: not this warp's to tell).
template <int NS>
__device__ __forceinline__ bool receive_unit(const Args<NS>& a, Bars* bars, uint32_t& q, int lane, Unit* u, uint32_t taken = 0) {
  for (;; ++q) {
    const uint32_t slot = q % kSched;
    if (!wait(&bars->sched_full[slot], (q / kSched) & 1, bars, a.st, 51)) return false;
    const int x = *reinterpret_cast<volatile int*>(&bars->sched_unit[slot]);
    if (x < a.n_units) *u = bars->sched_u[slot];
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->sched_empty[slot]);
    if (x >= a.n_units || bars->abort_flag) return false;
    if (taken != 0 && lane == 0) mbar_arrive_remote(taken);
    if (u->cnt != kBadList && u->cnt != kEmptyUnit) { ++q; return true; }
  }
}

// ---------------------------------------------------------------- softmax
// 32 columns of a row; `last` is the last one that the row sees
__device__ __forceinline__ void mask32(uint32_t* v, int last) {
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = i > last ? 0xff800000u : v[i];
}
__device__ __forceinline__ float max32(const uint32_t* v) {
  auto s = [&](int i) { return __uint_as_float(v[i]); };
  float mx0 = s(0), mx1 = s(1), mx2 = s(2), mx3 = s(3);
#pragma unroll
  for (int i = 4; i < 28; i += 8) {
    mx0 = max3(mx0, s(i), s(i + 1)); mx1 = max3(mx1, s(i + 2), s(i + 3));
    mx2 = max3(mx2, s(i + 4), s(i + 5)); mx3 = max3(mx3, s(i + 6), s(i + 7));
  }
  return fmaxf(max3(mx0, s(28), s(29)), max3(max3(mx1, s(30), s(31)), mx2, mx3));
}
// 32 probabilities of a row, to tensor memory; kEmul: every kEmulEvery-th pair of an unmasked tile on the FMA pipes
template <bool kF16, bool kEmul>
__device__ __forceinline__ void probabilities(const uint32_t* v, uint32_t dst, float c, float neg_mc, bool masked, float2& sum2) {
  const float2 c2 = make_float2(c, c), nm2 = make_float2(neg_mc, neg_mc);
  uint32_t pk[16];
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    const float2 xx = __ffma2_rn(make_float2(__uint_as_float(v[i]), __uint_as_float(v[i + 1])), c2, nm2);
    float2 p;
    if (kEmul && kEmulEvery > 0 && (i >> 1) % kEmulEvery == kEmulEvery - 1 && !masked) { p = exp2_poly2(xx); }
    else { p.x = ex2(xx.x); p.y = ex2(xx.y); }
    sum2 = __fadd2_rn(sum2, p);
    pk[i >> 1] = pack2<kF16>(p.x, p.y);
  }
  tmem_st16(dst, pk);
}

// S is read twice, 32 columns at a time with the next ones on their way: for the maximum, and for the exponentials, whose P goes over
// the first half of S.  Rolled up like this the code that a tile runs through stays small: the schedulers of an SM fetch
// instructions for six roles, and with a row of S in registers and everything unrolled the MMA warp, which passes its code once per
// tile, spent more time on fetching than on issuing (8192 tokens, 32 / 8 heads, segment 512, block 32, budget 1024: 131 -> 119 us; 111 us
// with waits and masks out of the way as well).
template <bool kF16, bool kEmul, int NS>
__device__ __forceinline__ void softmax_role(const Args<NS>& a, Bars* bars, float* stat, float2* sums, int rank, int wg, int warp, int lane) {
  const uint32_t tm = bars->tmem_base + (uint32_t(warp * 32) << 16);
  const uint32_t tO = tm + 384;
  const int row = warp * 32 + lane;
  const float c = a.sm_scale * 1.4426950408889634f;   // logits -> log2 units
  const uint32_t p_full = first_cta(bars->p_full);
  uint32_t g0 = 0;                                    // K/V tiles of the units before (all units)
  uint32_t un = 0;                                    // units before
  uint32_t q = 0;
  Unit u;
  while (receive_unit(a, bars, q, lane, &u)) {
    if (u.cnt == kZeroUnit) continue;
    const int mine = rank == 0 ? u.nA : u.nB;         // tiles that this CTA's rows see: none, or all but the last, or all

    for (int jt = int((g0 ^ uint32_t(wg)) & 1); jt < u.T; jt += 2) {
      const uint32_t g = g0 + jt, buf = g % kSlots;
      const uint32_t tS = tm + buf * 128;
      if (!wait(&bars->s_full[buf], (g / kSlots) & 1, bars, a.st, 10 + wg)) return;
      tc_fence_after();
      const bool seen = jt < mine;
      bool masked = false;
      int last[4];                                    // last visible column, counted from the first of each 32
      float m_tile = -CUDART_INF_F;
      uint32_t va[32], vb[32];
      const uint2 ref = row_load(&bars->ref[wg ^ 1][row]);
      if (seen) {
        if (u.generic) {
          // 128/blk listed blocks: a key counts iff its token is not after the row's (-1: none, also beyond the list)
          masked = true;
          const int bpt = kTile / a.blk, t = u.q_tok + rank * kTile + row;
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int li = jt * bpt + x * 32 / a.blk;
            last[x] = li < u.cnt ? t - __ldg(u.list + li) * a.blk - x * 32 % a.blk : -1;
          }
        } else {
          const bool diagonal = jt == mine - 1;
          masked = diagonal || (jt == u.n_past_tiles - 1 && u.last_cols < kTile);
#pragma unroll
          for (int x = 0; x < 4; ++x) last[x] = (diagonal ? row : u.last_cols - 1) - x * 32;
        }
        tmem_ld32(tS, va);
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
          tmem_wait_ld32(va);
          tmem_ld32(tS + x * 64 + 32, vb);
          if (CP_UNLIKELY(masked)) mask32(va, x ? last[2] : last[0]);
          m_tile = fmaxf(m_tile, max32(va));
          tmem_wait_ld32(vb);
          if (x == 0) tmem_ld32(tS + 64, va);
          if (CP_UNLIKELY(masked)) mask32(vb, x ? last[3] : last[1]);
          m_tile = fmaxf(m_tile, max32(vb));
        }
      }
      float m_prev = -CUDART_INF_F;
      if (g > 0) {
        if (!row_get(&bars->ref[wg ^ 1][row], ref, g, &m_prev, bars, a.st, 12 + wg)) return;
        if (jt == 0) m_prev = -CUDART_INF_F;
      }
      const float m_new = fmaxf(m_prev, m_tile);
      // lazy rescale: keep the old reference maximum while the new one exceeds it by < 2^8
      const bool need = jt > 0 && (m_new - m_prev) * c > kRescaleThreshold;
      const float m_run = (jt == 0 || need) ? m_new : m_prev;
      const float f = need ? ex2((m_prev - m_run) * c) : 1.f;
      row_put(&bars->ref[wg][row], m_run, g + 1);
      float2 sum2 = make_float2(0.f, 0.f);
      if (seen) {
        const float neg_mc = (m_run == -CUDART_INF_F) ? 0.f : -m_run * c;   // a row that has not seen a key yet (generic lists only): exp2(-inf) = 0
        tmem_ld32(tS, va);
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
          tmem_wait_ld32(va);
          tmem_ld32(tS + x * 64 + 32, vb);
          if (CP_UNLIKELY(masked)) mask32(va, x ? last[2] : last[0]);
          probabilities<kF16, kEmul>(va, tS + x * 32, c, neg_mc, masked, sum2);
          tmem_wait_ld32(vb);
          if (x == 0) tmem_ld32(tS + 64, va);
          if (CP_UNLIKELY(masked)) mask32(vb, x ? last[3] : last[1]);
          probabilities<kF16, kEmul>(vb, tS + x * 32 + 16, c, neg_mc, masked, sum2);
        }
        if (CP_UNLIKELY(__any_sync(0xffffffffu, need))) {
          // every P V up to the tile before must have gone into O; the next one waits for this warp
          if (!wait(&bars->v_empty[(g - 1) % kSlots], ((g - 1) / kSlots) & 1, bars, a.st, 14 + wg)) return;
          tc_fence_after();
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) {
            uint32_t ov[32];
            tmem_ld32(tO + qq * 32, ov);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * f);
            tmem_st32(tO + qq * 32, ov);
          }
        }
      }
      // what the tile adds to the row's sum, for the epilogue warp, which adds the tiles up in their order (handed from warpgroup to
      // warpgroup like the maximum, the sum made each wait for the other's P: 5 % at 8192 tokens)
      if (CP_UNLIKELY(g >= uint32_t(kSums) && int32_t(bars->added[warp] + kSums - 1 - g) < 0) && !wait_added(bars, warp, g - (kSums - 1), a.st)) return;
      sums[(g % kSums) * kTile + row] = make_float2(__fadd_rn(sum2.x, sum2.y), f);
      if (jt == u.T - 1) stat[(un % kSched) * kTile + row] = m_run;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_remote(p_full + buf * 8);
        mbar_arrive(&bars->sum_full[g % kSums][warp]);
      }
    }
    ++un;
    g0 += u.T;
  }
}

// ---------------------------------------------------------------- epilogue
// A warp's 32 rows: O / l, rounded, to shared memory (128-byte swizzle), and out by TMA, which drops rows beyond the sequence.
template <bool kF16, int NS>
__device__ __forceinline__ void epilogue_role(const Args<NS>& a, const OMaps<NS>& maps, Bars* bars, const float* stat, const float2* sums, uint32_t smem_base, int rank,
                                              int warp, int lane) {
  const uint32_t tO = bars->tmem_base + (uint32_t(warp * 32) << 16) + 384;
  const int row = warp * 32 + lane;
  const uint32_t o_empty = first_cta(&bars->o_empty);
  const uint32_t stage = smem_base + kSmemO + warp * 8192;      // two halves of [32 rows x 64 channels]
  uint32_t un = 0, q = 0, g = 0;
  Unit u;
  while (receive_unit(a, bars, q, lane, &u)) {
    const int t = u.q_tok + rank * kTile + row;
    if (u.cnt == kZeroUnit) {
      write_zero_row<128>(a, u, rank, t);
      continue;
    }
    float l = 0.f;
    bool ok = true;
    for (int jt = 0; jt < u.T && ok; ++jt, ++g) {
      ok = wait(&bars->sum_full[g % kSums][warp], (g / kSums) & 1, bars, a.st, 20);
      const float2 sf = sums[(g % kSums) * kTile + row];
      l = jt == 0 ? sf.x : __fadd_rn(__fmul_rn(l, sf.y), sf.x);
      __syncwarp();
      if (lane == 0) bars->added[warp] = g + 1;
    }
    if (!ok) break;
    const float m = stat[(un % kSched) * kTile + row];
    const float inv = l > 0.f ? 1.f / l : 0.f;                  // a row without any visible key (generic lists only): zeros
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");    // the rows of the unit before have left
    if (!wait(&bars->o_full, un & 1, bars, a.st, 21)) break;
    ++un;
    __syncwarp();
    tc_fence_after();
#pragma unroll
    for (int qq = 0; qq < 4; ++qq) {
      uint32_t ov[32];
      tmem_ld32(tO + qq * 32, ov);
      tmem_wait_ld();
      if (qq == 3) {                                            // O is read: the next unit's P V may overwrite it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(o_empty);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {                             // 16-byte chunks (qq & 1) * 4 + i of half qq >> 1
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          w[e] = pack2<kF16>(__uint_as_float(ov[8 * i + 2 * e]) * inv, __uint_as_float(ov[8 * i + 2 * e + 1]) * inv);
        const uint32_t dst = stage + (qq >> 1) * 4096 + lane * 128 + ((((qq & 1) * 4 + i) ^ (lane & 7)) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    const int t0 = u.q_tok + rank * kTile + warp * 32;
    if (lane == 0 && (rank == 0 || u.rowsB) && t0 < u.n) {
      const CUtensorMap* tm = maps.m + (NS > 1 ? u.seq : 0);
      tma_store_4d(tm, stage, 0, t0, u.h, u.b);
      tma_store_4d(tm, stage + 4096, 64, t0, u.h, u.b);
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    if (a.lse != nullptr && (rank == 0 || u.rowsB) && t < u.n)
      a.lse[a.seq[u.seq].lse0 + ((long long)u.b * a.Hq + u.h) * u.n + t] = m * a.sm_scale + __logf(l);
  }
  if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------- producers
// Each CTA brings in its own rows of Q, its 64 keys of a K tile and its 64 channels of a V tile; the bytes of both CTAs are counted
// by the first CTA's barriers.  One lane per box of a gathered tile; boxes beyond the list read past the end of the tensor and
// arrive as zeros.
template <int NS>
__device__ __forceinline__ void producer_k_role(const Args<NS>& a, const Maps<NS>& maps, Bars* bars, uint32_t smem_base, int rank, int lane) {
  const int bpt = kTile / a.blk, rows = min(a.blk, 64), nb = 64 / rows;    // boxes of 64 keys: nb blocks (or half a block), two halves of channels
  const int my_blk = lane >> 1, my_hf = lane & 1;
  const uint32_t k_full = first_cta(bars->k_full), q_full = first_cta(bars->q_full), taken = first_cta(&bars->taken);
  uint32_t g = 0, un = 0, q = 0;
  Unit u;
  while (receive_unit(a, bars, q, lane, &u, taken)) {
    if (u.cnt == kZeroUnit) continue;
    const CUtensorMap* tm = maps.m[NS > 1 ? u.seq : 0];
    auto token_of = [&](int jt) {
      const int li = jt * bpt + (a.blk == 128 ? 0 : rank * nb) + my_blk;
      return my_blk < nb && jt < u.n_past_tiles && li < u.n_past ? u.list[li] * a.blk + (a.blk == 128 ? rank * 64 : 0) : u.n;
    };
    int tok = token_of(0);
    const uint32_t qb = un & 1;
    if (un >= 2 && !wait(&bars->q_empty[qb], ((un >> 1) - 1) & 1, bars, a.st, 31)) return;
    if (lane == 0 && rank == 0) mbar_expect_tx(&bars->q_full[qb], 2 * kQBytes);
    __syncwarp();
    if (lane < 2) tma_load_pair(smem_base + kSmemQ + qb * kQBytes + lane * kHalfBytes, tm + kQ, q_full + qb * 8, lane * 64, u.q_tok + rank * kTile, u.h, u.b);
    ++un;
    for (int jt = 0; jt < u.T; ++jt, ++g) {
      const uint32_t slot = g % kSlots;
      const int next_tok = token_of(jt + 1);            // the next tile's list entries are on their way during the wait
      if (g >= kSlots && !wait(&bars->s_full[slot], (g / kSlots - 1) & 1, bars, a.st, 30)) return;
      if (lane == 0 && rank == 0) mbar_expect_tx(&bars->k_full[slot], 2 * kSlotBytes);
      __syncwarp();
      const uint32_t dst = smem_base + kSmemK + slot * kSlotBytes + my_hf * (kSlotBytes / 2);
      if (jt < u.n_past_tiles) {
        if (my_blk < nb) tma_load_pair(dst + my_blk * rows * 128, tm + kKb, k_full + slot * 8, my_hf * 64, tok, u.kvh, u.b);
      } else if (lane < 2) {
        const int ci = jt - u.n_past_tiles;
        const int t0 = ci < u.n_cont ? u.c_tok + ci * kTile : u.d_tok + (ci - u.n_cont) * kTile;
        tma_load_pair(dst, tm + kKt, k_full + slot * 8, my_hf * 64, t0 + rank * 64, u.kvh, u.b);
      }
      __syncwarp();
      tok = next_tok;
    }
  }
}
template <int NS>
__device__ __forceinline__ void producer_v_role(const Args<NS>& a, const Maps<NS>& maps, Bars* bars, uint32_t smem_base, int rank, int lane) {
  const int bpt = kTile / a.blk;
  const uint32_t v_full = first_cta(bars->v_full);
  uint32_t g = 0, q = 0;
  Unit u;
  while (receive_unit(a, bars, q, lane, &u)) {
    if (u.cnt == kZeroUnit) continue;
    const CUtensorMap* tm = maps.m[NS > 1 ? u.seq : 0];
    auto token_of = [&](int jt) {
      const int li = jt * bpt + lane;
      return lane < bpt && jt < u.n_past_tiles && li < u.n_past ? u.list[li] * a.blk : u.n;
    };
    int tok = token_of(0);
    for (int jt = 0; jt < u.T; ++jt, ++g) {
      const uint32_t slot = g % kSlots;
      const int next_tok = token_of(jt + 1);
      if (g >= kSlots && !wait(&bars->v_empty[slot], (g / kSlots - 1) & 1, bars, a.st, 32)) return;
      if (!a.withhold_v) {
        if (lane == 0 && rank == 0) mbar_expect_tx(&bars->v_full[slot], 2 * kSlotBytes);
        __syncwarp();
        const uint32_t dst = smem_base + kSmemV + slot * kSlotBytes;
        if (jt < u.n_past_tiles) {
          if (lane < bpt) tma_load_pair(dst + lane * a.blk * 128, tm + kVb, v_full + slot * 8, rank * 64, tok, u.kvh, u.b);
        } else if (lane == 0) {
          const int ci = jt - u.n_past_tiles;
          const int t0 = ci < u.n_cont ? u.c_tok + ci * kTile : u.d_tok + (ci - u.n_cont) * kTile;
          tma_load_pair(dst, tm + kVt, v_full + slot * 8, rank * 64, t0, u.kvh, u.b);
        }
      }
      __syncwarp();
      tok = next_tok;
    }
  }
}

// ---------------------------------------------------------------- MMA issuer (first CTA)
// S(g) goes to buffer g % 3 as soon as P V of tile g - 3 has been issued (MMAs run in the order of issue), so up to three tiles ahead
// and on into the next units; P V follows as the tiles' P arrive.  At the end of a unit the next one is begun early if it has been drawn.
// Sixteen MMAs run for 1040 cycles, and what this warp executes besides issuing them must stay far below that, so P V of a tile and QK^T
// of the tile three ahead are issued together, behind one set of waits.
template <bool kF16, int NS>
__device__ __forceinline__ void mma_role(const Args<NS>& a, Bars* bars, uint32_t smem_base, int lane) {
  const uint32_t tm = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  const uint32_t tO = tm + 384;
  const uint64_t desc = desc_base(16);    // all operands are one 128-byte swizzled atom wide: no leading-dimension offset
  uint32_t q = 0;                         // units received
  uint32_t gq = 0, gp = 0;                // tiles whose QK^T / P V have been issued
  uint32_t uq = 0, up = 0;                // units with tiles that QK^T has begun / P V has finished
  uint32_t info = 0;                      // of the unit that P V is in (mma_unit)
  int jq = 0, Tq = 0, jp = 0;             // tile within its unit: QK^T, its unit's tiles, P V
  bool end = false;
  // QK^T of as many tiles as S has room for, the next unit's too; waits for that unit only if there is nothing else to do
  auto advance = [&]() {
    while (!end && gq < gp + 3) {
      if (jq == Tq) {
        const uint32_t slot = q % kSched;
        if (gq != gp && !__any_sync(0xffffffffu, mbar_test(&bars->sched_full[slot], (q / kSched) & 1))) return true;
        if (!wait(&bars->sched_full[slot], (q / kSched) & 1, bars, a.st, 51)) return false;
        const int x = *reinterpret_cast<volatile int*>(&bars->sched_unit[slot]);
        const Unit* su = &bars->sched_u[slot];
        const int cnt = x < a.n_units ? su->cnt : kEmptyUnit;
        const int T = su->T;
        const uint32_t second = su->nB > su->nA ? 0x80000000u : 0u;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->sched_empty[slot]);
        ++q;
        if (bars->abort_flag) return false;
        if (x >= a.n_units) { end = true; return true; }
        if (cnt == kBadList || cnt == kEmptyUnit || cnt == kZeroUnit) continue;
        if (lane == 0) bars->mma_unit[uq & 3] = uint32_t(T) | second;
        __syncwarp();
        Tq = T; jq = 0;
        if (!wait(&bars->q_full[uq & 1], (uq >> 1) & 1, bars, a.st, 41)) return false;
        ++uq;
      }
      const uint32_t slot = gq % kSlots;
      if (!wait(&bars->k_full[slot], (gq / kSlots) & 1, bars, a.st, 40)) return false;
      __syncwarp();
      umma2_qk8(tm + slot * 128, desc_at(desc, smem_base + kSmemQ + ((uq - 1) & 1) * kQBytes), desc_at(desc, smem_base + kSmemK + slot * kSlotBytes),
                Idesc2<kF16>::qk);
      umma2_commit(&bars->s_full[slot]);
      ++gq;
      if (++jq == Tq) umma2_commit(&bars->q_empty[(uq - 1) & 1]);   // that was the unit's last QK^T: Q may be replaced
    }
    return true;
  };
  uint32_t slot = 0, par = 0;             // of tile gp, and the parity of its phase
  bool v_ok = false, k_ok = false;        // the V tile of gp, and the K tile three ahead, are known to have arrived
  for (;;) {
    if (CP_UNLIKELY(gq != gp + 3)) {                   // the start, and the end of a unit whose successor has not been drawn in time
      if (!advance()) return;
      if (gp == gq) {
        if (end) return;
        continue;
      }
    }
    if (CP_UNLIKELY(jp == 0)) {
      info = *reinterpret_cast<volatile uint32_t*>(&bars->mma_unit[up & 3]);
      if (up > 0 && !wait(&bars->o_empty, (up - 1) & 1, bars, a.st, 44)) return;
    }
    const bool next = gq == gp + 3 && jq < Tq;   // the tile three ahead is of a unit that QK^T is in: it follows in the same breath
    const bool last = jp == int(info & 0x7fffffffu) - 1;
    const uint64_t dv = desc_at(desc, smem_base + kSmemV + slot * kSlotBytes), dk = desc_at(desc, smem_base + kSmemK + slot * kSlotBytes);
    const uint64_t dq = desc_at(desc, smem_base + kSmemQ + ((uq - 1) & 1) * kQBytes);
    const uint32_t tP = tm + slot * 128;
    if (CP_UNLIKELY(!v_ok) && !wait_slow(&bars->v_full[slot], par, bars, a.st, 45)) return;
    if (CP_UNLIKELY(next && !k_ok) && !wait_slow(&bars->k_full[slot], par ^ 1, bars, a.st, 40)) return;
    const uint32_t slot1 = slot == kSlots - 1 ? 0 : slot + 1, par1 = par ^ (slot == kSlots - 1 ? 1u : 0u);   // of the next tile
    if (CP_UNLIKELY(!wait(&bars->p_full[slot], par, bars, a.st, 42))) return;
    __syncwarp();
    tc_fence_after();
    if (CP_UNLIKELY(last && (info >> 31))) {
#pragma unroll 1
      for (int kk = 0; kk < 8; ++kk) umma2_ts_second(tO, tP + kk * 8, dv + kk * 128, Idesc2<kF16>::pv);
    } else {
      umma2_pv8(tO, tP, dv, Idesc2<kF16>::pv, jp > 0 ? 1u : 0u);
    }
    umma2_commit(&bars->v_empty[slot]);
    // under the MMAs just issued: what the next turn would wait for
    v_ok = mbar_ready(&bars->v_full[slot1], par1);
    k_ok = gq != gp + 1 && mbar_ready(&bars->k_full[slot1], par1 ^ 1);
    if (CP_LIKELY(next)) {
      umma2_qk8(tP, dq, dk, Idesc2<kF16>::qk);
      umma2_commit(&bars->s_full[slot]);
      ++gq;
      if (CP_UNLIKELY(++jq == Tq)) umma2_commit(&bars->q_empty[(uq - 1) & 1]);
    }
    ++gp;
    ++jp;
    if (CP_UNLIKELY(last)) {
      umma2_commit(&bars->o_full);
      ++up;
      jp = 0;
    }
    slot = slot1;
    par = par1;
  }
}

// ---------------------------------------------------------------- kernel
template <bool kF16, bool kEmul, int NS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
attention_pair_kernel(const __grid_constant__ Maps<NS> maps, const __grid_constant__ OMaps<NS> o_maps, const __grid_constant__ Args<NS> a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t smem_base = (raw + 1023u) & ~1023u;       // the same in both CTAs
  uint8_t* smem = smem_raw + (smem_base - raw);
  Bars* bars = reinterpret_cast<Bars*>(smem + kSmemBar);
  float* stat = reinterpret_cast<float*>(smem + kSmemStat);
  float2* sums = reinterpret_cast<float2*>(smem + kSmemSum);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = int(blockIdx.x & 1);

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->q_full[i], 1); mbar_init(&bars->q_empty[i], 1); }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&bars->k_full[i], 1); mbar_init(&bars->v_full[i], 1); mbar_init(&bars->v_empty[i], 1); mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->p_full[i], 8);                  // 4 warps of each CTA
    }
    mbar_init(&bars->o_full, 1);
    mbar_init(&bars->o_empty, 8);
    for (int i = 0; i < kSched; ++i) {
      mbar_init(&bars->sched_full[i], 1);
      mbar_init(&bars->sched_empty[i], kReaders - (rank == 0 ? 0 : 1));   // the MMA warp is the first CTA's
    }
    for (int i = 0; i < kSums * 4; ++i) mbar_init(&bars->sum_full[i >> 2][i & 3], 1);
    for (int i = 0; i < 4; ++i) bars->added[i] = 0;
    mbar_init(&bars->clc_full, 1);
    mbar_init(&bars->taken, 2);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp < 8) bars->ref[warp >> 2][threadIdx.x & 127] = 0ull;
  if (warp == 12 && lane < kMaps && NS == 1) prefetch_tmap(&maps.m[0][lane]);
  if (warp == 14) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&bars->tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  pdl_wait();

  if (warp < 8) {
    softmax_role<kF16, kEmul, NS>(a, bars, stat, sums, rank, warp >> 2, warp & 3, lane);
  } else if (warp < 12) {
    epilogue_role<kF16, NS>(a, o_maps, bars, stat, sums, smem_base, rank, warp & 3, lane);
  } else {
    if (warp == 12) producer_k_role<NS>(a, maps, bars, smem_base, rank, lane);
    else if (warp == 13) producer_v_role<NS>(a, maps, bars, smem_base, rank, lane);
    else if (warp == 14) { if (rank == 0) mma_role<kF16, NS>(a, bars, smem_base, lane); }
    else scheduler_role<NS>(a, bars, rank, lane);
  }
  if (bars->abort_flag) {
    // give copies and MMAs still in flight time to land before the CTA's resources go away
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                          // neither CTA leaves while the other may read its operands or arrive at its barriers
  if (warp == 14) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(bars->tmem_base) : "memory");
}

template <bool kF16, bool kEmul, int NS>
int launch_variant(const Maps<NS>& maps, const OMaps<NS>& o_maps, const Args<NS>& a, cudaStream_t s) {
  auto kern = attention_pair_kernel<kF16, kEmul, NS>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal) != cudaSuccess) return CP_ERR_CUDA;
  return launch_pdl(kern, dim3(unsigned(a.n_units) * 2), kThreads, kSmemTotal, s, maps, o_maps, a);   // the cluster size is the kernel's own
}
}  // namespace

template <int NS>
int launch_attention_pair(const Maps<NS>& maps, const OMaps<NS>& o_maps, const Args<NS>& a, bool f16, cudaStream_t s) {
  if (a.emul) return f16 ? launch_variant<true, true, NS>(maps, o_maps, a, s) : launch_variant<false, true, NS>(maps, o_maps, a, s);
  return f16 ? launch_variant<true, false, NS>(maps, o_maps, a, s) : launch_variant<false, false, NS>(maps, o_maps, a, s);
}
template int launch_attention_pair<1>(const Maps<1>&, const OMaps<1>&, const Args<1>&, bool, cudaStream_t);
template int launch_attention_pair<kMaxSeqs>(const Maps<kMaxSeqs>&, const OMaps<kMaxSeqs>&, const Args<kMaxSeqs>&, bool, cudaStream_t);

}  // namespace cp
