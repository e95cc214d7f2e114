// K4 / K5: block-sparse (Algorithm 2, lines 6-13) and dense causal (Eq. 2) attention on the
// sm_100a tensor cores.  bf16 or fp16 operands, head_dim 128 or 64, fp32 accumulation in tensor memory, online softmax.
//
// CTAs (one per SM) walk over work units; a unit is 256 consecutive query rows of one
// (batch, query head): two 128-row tiles "A" and "B" that share every K/V tile the producer brings in
// (tile B is absent in the last unit of a segment with an odd number of 128-row tiles).  Roles (384 threads):
//   warps 0-3  softmax for tile A (one thread per query row)
//   warps 4-7  softmax for tile B
//   warp  8    TMA producer: K/V tiles through a ring of 5 x 32 KB (head_dim 64: 8 x 16 KB); a gathered
//              tile is assembled from 128/blk boxes addressed by the block list
//   warp  9    MMA issuer: S = Q K^T (operands in shared memory), O += P V (P read from tensor
//              memory, where the softmax warps overwrite S with 16-bit probabilities)
//   warp  10   scheduler: draws the next unit, reads and checks its block list, publishes it
//              (warp 11 is idle; it completes the third warpgroup)
// Tensor memory (512 columns): S_A | S_B (128 fp32 columns each) | O_A | O_B (head_dim columns each) | head_dim 64 in bf16: the third
// parts of P_A | P_B (64 columns each).
// The tile sequence of a unit is: gathered past tiles, contiguous unmasked tiles, then the
// diagonal tiles; tile A stops one tile earlier than B.  The grid has one CTA per unit; those that
// are resident take over the units of those that have not started yet, one after another
// (clusterlaunchcontrol.try_cancel, scheduler warp), and publish them to the other warps, so faster SMs
// take more units without a counter in memory that a launch of its own would have to clear (and whose
// round trip had to be waited out).  With the scheduler warp and the order of units below, against a counter that the producer
// warp read, 32 heads, segment 512, block 32, budget 1024, medians of nine: 1300 tokens 47.3 -> 32.4 us, 8192 145 -> 128, 131072
// 2234 -> 2110 us; dense 4096 tokens 176 -> 141 us, 20001 unchanged (3.0 ms).  Every wait is bounded: on expiry the waiter raises a CTA-wide abort flag and CP_ERR_TIMEOUT, and all roles drain.
// One launch serves one problem or a packed batch of up to kMaxSeqs sequences (each with tensor maps of
// its own, so that reads past a sequence's end arrive as zeros and never as a neighbour's tokens).
#include <algorithm>

#include "attention_units.cuh"

namespace cp {
namespace {

constexpr int kThreads = 384;   // 3 warpgroups: softmax A, softmax B, {producer, MMA, scheduler, idle}
constexpr int kMaxSlots = 8;
constexpr int kBarBytes = 512;
// What head_dim decides.  Heads of 64 channels keep 32-bit probabilities and sums (softmax_role64): P goes to the tensor cores as a
// sum of 16-bit values of its own, two in fp16 (22 bits) and three in bf16 (24 bits), O += P V runs over each of them, and the
// 64 columns of a tile's P V are added up in registers, because the tensor cores round every accumulation towards zero.
// Tensor memory then holds, besides S, a tile's P V of each query tile and the third part of P (64 columns each).
template <int D> struct Shape {
  static constexpr bool kSplitP = D == 64;                          // see above
  static constexpr int kHalves = D / 64;
  static constexpr int kTileBytes = kHalves * kHalfBytes;
  static constexpr int kSlots = D == 128 ? 5 : kMaxSlots;           // 5 x 32 KB + 64 KB of Q; 8 x 16 KB + 32 KB
  static constexpr int kSmemQ = 0;
  static constexpr int kSmemKV = 2 * kTileBytes;
  static constexpr int kSmemBar = kSmemKV + kSlots * kTileBytes;
  static constexpr int kSmemTotal = kSmemBar + kBarBytes + 1024;    // + barrier block + slack to align the tiles to 1024 bytes
};
// fp16 parts of P are scaled by 2^7: the reference maximum is at most 2^8 behind (lazy rescale), so P stays below 2^15,
// and the low parts of small probabilities stay out of the subnormals
template <bool kF16> constexpr float kPShift = kF16 ? 7.f : 0.f;
constexpr int kRegPoolNeeded = 256 * 216 + 128 * 64;   // registers the roles hold after setmaxnreg (softmax 216, producer/MMA 64)

struct Bars {
  unsigned long long q_full;
  unsigned long long q_empty;
  unsigned long long kv_full[kMaxSlots];
  unsigned long long kv_empty[kMaxSlots];
  unsigned long long s_full[2];
  unsigned long long p_full[2];
  unsigned long long o_done[2];
  unsigned long long sched_full[2];
  unsigned long long sched_empty[2];
  unsigned long long clc_full;
  unsigned long long taken;            // the producer has begun the unit published last: the next one may be drawn
  __align__(16) uint32_t clc_resp[4];  // the hardware's answer to the last request for a further unit
  int sched_unit[2];
  Unit sched_u[2];                   // the published unit, decoded; its cnt carries kBadList / kEmptyUnit
  uint32_t tmem_base;
  volatile int abort_flag;
  volatile uint32_t beat;            // advanced by warps that evaluate rows one by one (exact_row)
};

// bounded wait on one of this kernel's barriers (the CTA's abort flag lives in the barrier block)
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity, Bars* bars, DeviceStatus* st, int site) {
  return mbar_wait(bar, parity, &bars->abort_flag, st, site, &bars->beat);
}

// ---------------------------------------------------------------- unit scheduler
// The scheduler warp gets the q-th unit of this CTA (its own block index first, then those of CTAs that the hardware
// lets it cancel), reads and checks its block list, and publishes (unit, list length) through a two-entry ring; the
// other warps take it from there and touch no global memory at a unit's start.  This is a chain of three round trips
// (3-4 K cycles): in the producer warp it held up the loads of the unit before (figures: head of this file).
// A unit is drawn when the producer begins the one before it, no earlier, so that no CTA sits on units at the end.
// A list that breaks its contract is published with length kBadList and skipped by everyone.
__device__ __forceinline__ void request_unit(Bars* bars) {
  mbar_expect_tx(&bars->clc_full, 16);
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
               ::"r"(smem_u32(bars->clc_resp)), "r"(smem_u32(&bars->clc_full)) : "memory");
}
// block index of the cancelled CTA, or `none` when every CTA has started (no further request may be made then)
__device__ __forceinline__ int requested_unit(Bars* bars, int none) {
  uint32_t ok, x;
  asm volatile(
      "{\n.reg .pred p;\n.reg .b128 r;\nld.shared.b128 r, [%2];\n"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\nselp.u32 %0, 1, 0, p;\nmov.u32 %1, 0;\n"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, _, _, _}, r;\n}"
      : "=r"(ok), "=r"(x) : "r"(smem_u32(bars->clc_resp)) : "memory");
  return ok ? int(x) : none;
}
template <int NS>
__device__ __forceinline__ void scheduler_role(const Args<NS>& a, Bars* bars, int lane) {
  for (uint32_t q = 0;; ++q) {
    const uint32_t slot = q & 1;
    if (q >= 2 && !mbar_wait(&bars->sched_empty[slot], ((q >> 1) - 1) & 1, bars, a.st, 50)) return;
    int x = int(blockIdx.x);
    if (q > 0) {
      if (!mbar_wait(&bars->taken, (q - 1) & 1, bars, a.st, 53)) return;
      __syncwarp();
      if (lane == 0) request_unit(bars);
      if (!mbar_wait(&bars->clc_full, (q - 1) & 1, bars, a.st, 52)) return;
      x = requested_unit(bars, a.n_units);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the answer has been read before the next one is written
    }
    Unit u;
    int cnt = 0;
    if (x < a.n_units) {
      u = decode_unit(a, x, kLoadCnt);
      cnt = u.cnt;
      if (u.q_tok >= u.n) {
        cnt = kEmptyUnit;                               // a short last segment has fewer units
      } else {
        const int cls = classify_unit(a, u, lane);
        if (cls < 0) {
          if (lane == 0) report(a.st, CP_ERR_BOUNDS, 1, u.b, u.h, u.seg_j, u.cnt);
          cnt = kBadList;
        } else if (cls == 1) {
          // any other valid list: all listed blocks are gathered, both query tiles consume every tile
          u.generic = 1;
          u.n_past = cnt;
          u.n_past_tiles = (cnt * a.blk + kTile - 1) / kTile;
          u.last_cols = cnt * a.blk - (u.n_past_tiles - 1) * kTile;
          u.n_cont = 0;
          u.nA = u.n_past_tiles;
          u.nB = u.rowsB ? u.n_past_tiles : 0;
          u.T = u.n_past_tiles;
          if (u.T == 0) cnt = kZeroUnit;           // nothing listed: the rows are zeros
        }
      }
    }
    u.cnt = cnt;
    if (lane == 0) {
      bars->sched_unit[slot] = x;
      if (x < a.n_units) bars->sched_u[slot] = u;
      mbar_arrive(&bars->sched_full[slot]);
    }
    if (x >= a.n_units) return;
    // Only this warp reads the status word in global memory (a round trip the other roles would otherwise
    // pay at every unit); it tells them through the CTA's abort flag, which their waits poll.
    if (stop_requested(a, bars)) { bars->abort_flag = 1; return; }
  }
}
template <int NS>
__device__ __forceinline__ bool receive_unit(const Args<NS>& a, Bars* bars, uint32_t q, int lane, int* x_out, Unit* u_out) {
  const uint32_t slot = q & 1;
  if (!mbar_wait(&bars->sched_full[slot], (q >> 1) & 1, bars, a.st, 51)) return false;
  *x_out = *reinterpret_cast<volatile int*>(&bars->sched_unit[slot]);
  if (*x_out < a.n_units) *u_out = bars->sched_u[slot];
  else u_out->cnt = kEmptyUnit;
  __syncwarp();
  if (lane == 0) mbar_arrive(&bars->sched_empty[slot]);
  return true;
}

// ---------------------------------------------------------------- softmax role
constexpr int kMaskNone = 0, kMaskCausal = 1, kMaskCols = 2, kMaskGeneric = 3;
// One row of a 64-channel head by one warp over exactly the keys it sees, in plain fp32.  A tile's MMA multiplies the zero
// probability of a key that the row does not see with that key's value, which is NaN where the value is infinite or NaN; a row
// whose output came out as NaN or infinite is therefore evaluated again here.  A row of 131072 keys takes milliseconds and a unit
// has up to 256 of them, so the CTA's other warps are told that this one is at work (`beat`), and their waits go on.
template <bool kF16, int NS>
__device__ __noinline__ void exact_row(const Args<NS>* ap, Bars* bars, int seq, int b, int h, const int32_t* list, int cnt, int t, int lane) {
  const Args<NS>& a = *ap;
  const Seq& sq = a.seq[seq];
  const uint4* q4 = reinterpret_cast<const uint4*>(a.Q + b * a.qs[0] + h * a.qs[1] + (sq.tok0 + t) * a.qs[2]);
  const uint16_t* kb = a.K + b * a.ks[0] + (h / a.g) * a.ks[1] + sq.tok0 * a.ks[2];
  const uint16_t* vb = a.V + b * a.vs[0] + (h / a.g) * a.vs[1] + sq.tok0 * a.vs[2];
  const int n_ranges = a.dense ? 1 : cnt;
  float m_run = -CUDART_INF_F, l_run = 0.f;
  float2 acc = make_float2(0.f, 0.f);                       // channels 2 * lane, 2 * lane + 1
  uint32_t chunk = 0;
  for (int e = 0; e < n_ranges; ++e) {
    const int u0 = a.dense ? 0 : list[e] * a.blk, u1 = a.dense ? t + 1 : min(u0 + a.blk, t + 1);
    for (int base = u0; base < u1; base += 32) {
      if ((chunk++ & 63u) == 0 && lane == 0) bars->beat = bars->beat + 1;
      const int u = base + lane;
      float s = -CUDART_INF_F;
      if (u < u1) {
        const uint4* k4 = reinterpret_cast<const uint4*>(kb + int64_t(u) * a.ks[2]);
        float x = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint4 qw = q4[c], kw = k4[c];
          const uint32_t qe[4] = {qw.x, qw.y, qw.z, qw.w}, ke[4] = {kw.x, kw.y, kw.z, kw.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 qf = unpack2<kF16>(qe[i]), kf = unpack2<kF16>(ke[i]);
            x = fmaf(qf.y, kf.y, fmaf(qf.x, kf.x, x));
          }
        }
        s = x * a.sm_scale;
      }
      float mx = s;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(m_run, mx);
      const float corr = m_run == -CUDART_INF_F ? 0.f : expf(m_run - m_new);
      const float p = u < u1 ? expf(s - m_new) : 0.f;
      float ps = p;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
      l_run = l_run * corr + ps;
      m_run = m_new;
      acc.x *= corr; acc.y *= corr;
      const int here = min(32, u1 - base);
#pragma unroll 8
      for (int kk = 0; kk < here; ++kk) {
        const float pk = __shfl_sync(0xffffffffu, p, kk);
        const float2 vf = unpack2<kF16>(*reinterpret_cast<const uint32_t*>(vb + int64_t(base + kk) * a.vs[2] + 2 * lane));
        acc.x = fmaf(pk, vf.x, acc.x); acc.y = fmaf(pk, vf.y, acc.y);
      }
    }
  }
  const float inv = l_run > 0.f ? 1.f / l_run : 0.f;        // a row without any visible key: zeros, lse = ln 0
  uint16_t* o = a.O + b * a.osb + h * a.osh + (sq.tok0 + t) * a.ost;
  *reinterpret_cast<uint32_t*>(o + 2 * lane) = pack2<kF16>(acc.x * inv, acc.y * inv);
  if (a.lse != nullptr && lane == 0) a.lse[sq.lse0 + ((long long)b * a.Hq + h) * sq.n + t] = m_run + logf(l_run);
}

template <bool kF16, int NS>
__device__ __forceinline__ void softmax_role(const Args<NS>& a, Bars* bars, int which, int warp_in_wg, int lane) {
  constexpr int D = 128;
  const uint32_t tm = bars->tmem_base;
  const uint32_t lane_off = uint32_t(warp_in_wg * 32) << 16;
  const uint32_t tS = tm + lane_off + which * 128;
  const uint32_t tO = tm + lane_off + 256 + which * D;
  const int row = warp_in_wg * 32 + lane;
  const float c = a.sm_scale * 1.4426950408889634f;   // logits -> log2 units
  uint32_t n_tiles = 0;                               // S tiles consumed so far (all units)
  uint32_t n_units = 0;                               // units finished so far

  for (uint32_t q = 0;; ++q) {
    int x;
    Unit u;
    if (!receive_unit(a, bars, q, lane, &x, &u) || x >= a.n_units || bars->abort_flag) return;
    if (u.cnt == kBadList || u.cnt == kEmptyUnit) continue;
    if (u.cnt == kZeroUnit) {
      write_zero_row<D>(a, u, which, u.q_tok + which * kTile + row);
      continue;
    }
    const int my_tiles = which == 0 ? u.nA : u.nB;
    if (my_tiles == 0) continue;                        // this unit has no tile B
    float m_run = -CUDART_INF, l_run = 0.f;

    for (int jt = 0; jt < my_tiles; ++jt, ++n_tiles) {
      if (!mbar_wait(&bars->s_full[which], n_tiles & 1, bars, a.st, 10 + which)) return;
      tc_fence_after();
      uint32_t sv[128];
      tmem_ld128(tS, sv);
      tmem_wait_ld();
      float* s = reinterpret_cast<float*>(sv);

      int kind = kMaskNone, cols = kTile;
      if (u.generic) kind = kMaskGeneric;
      else if (jt == my_tiles - 1) kind = kMaskCausal;                              // own diagonal tile
      else if (jt == u.n_past_tiles - 1 && u.last_cols < kTile) { kind = kMaskCols; cols = u.last_cols; }
      if (kind == kMaskGeneric) {
        // a gathered tile of a generic list: the tile holds 128/blk listed blocks; key column i belongs to token
        // list[...]*blk + i % blk and counts iff that token is not after this row's token.  lim[q] = last visible
        // offset inside sub-block q (-1: none, also for sub-blocks beyond the list)
        const int t_row = u.q_tok + which * kTile + row;
        const int bpt = kTile / a.blk;
        int lim[4];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
          const int li = jt * bpt + qq;
          lim[qq] = (qq < bpt && li < u.cnt) ? t_row - __ldg(u.list + li) * a.blk : -1;
        }
        if (a.blk == 128) {
#pragma unroll
          for (int i = 0; i < 128; ++i) s[i] = (i > lim[0]) ? -CUDART_INF : s[i];
        } else if (a.blk == 64) {
#pragma unroll
          for (int i = 0; i < 128; ++i) s[i] = ((i & 63) > lim[i >> 6]) ? -CUDART_INF : s[i];
        } else {
#pragma unroll
          for (int i = 0; i < 128; ++i) s[i] = ((i & 31) > lim[i >> 5]) ? -CUDART_INF : s[i];
        }
      } else if (kind == kMaskCausal) {
#pragma unroll
        for (int i = 0; i < 128; ++i) s[i] = (i > row) ? -CUDART_INF : s[i];
      } else if (kind == kMaskCols) {
#pragma unroll
        for (int i = 0; i < 128; ++i) s[i] = (i >= cols) ? -CUDART_INF : s[i];
      }
      float mx0 = s[0], mx1 = s[1], mx2 = s[2], mx3 = s[3];
#pragma unroll
      for (int i = 4; i < 124; i += 8) {
        mx0 = max3(mx0, s[i], s[i + 1]); mx1 = max3(mx1, s[i + 2], s[i + 3]);
        mx2 = max3(mx2, s[i + 4], s[i + 5]); mx3 = max3(mx3, s[i + 6], s[i + 7]);
      }
      mx0 = max3(mx0, s[124], s[125]); mx1 = max3(mx1, s[126], s[127]);
      const float m_tile = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
      const float m_new = fmaxf(m_run, m_tile);
      // lazy rescale: keep the old reference maximum while the new one exceeds it by < 2^8
      const bool need = (m_new - m_run) * c > kRescaleThreshold;   // true on the first tile (m_run = -inf)
      if (jt == 0) {
        m_run = m_new;
      } else if (__any_sync(0xffffffffu, need)) {
        const float f = need ? ex2((m_run - m_new) * c) : 1.f;
        if (need) { m_run = m_new; l_run *= f; }
#pragma unroll
        for (int q = 0; q < D / 32; ++q) {
          uint32_t ov[32];
          tmem_ld32(tO + q * 32, ov);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * f);
          tmem_st32(tO + q * 32, ov);
        }
      }
      const float neg_mc = (m_run == -CUDART_INF) ? 0.f : -m_run * c;   // a row that has not seen a key yet (generic lists only): exp2(-inf) = 0
      const float2 c2 = make_float2(c, c), nm2 = make_float2(neg_mc, neg_mc);
      float2 sum2 = make_float2(0.f, 0.f);
      uint32_t pk[64];
      if (kind == kMaskNone && a.emul) {
        // unmasked tile of a long unit: every kEmulEvery-th pair takes the polynomial path, the rest the MUFU
#pragma unroll
        for (int i = 0; i < 128; i += 2) {
          const float2 xx = __ffma2_rn(make_float2(s[i], s[i + 1]), c2, nm2);
          float2 p;
          if (kEmulEvery > 0 && (i >> 1) % kEmulEvery == kEmulEvery - 1) { p = exp2_poly2(xx); }
          else { p.x = ex2(xx.x); p.y = ex2(xx.y); }
          sum2 = __fadd2_rn(sum2, p);
          pk[i >> 1] = pack2<kF16>(p.x, p.y);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 128; i += 2) {
          const float2 xx = __ffma2_rn(make_float2(s[i], s[i + 1]), c2, nm2);
          float2 p;
          p.x = ex2(xx.x); p.y = ex2(xx.y);
          sum2 = __fadd2_rn(sum2, p);
          pk[i >> 1] = pack2<kF16>(p.x, p.y);
        }
      }
      l_run += sum2.x + sum2.y;
      tmem_st64(tS, pk);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&bars->p_full[which]);
    }

    // epilogue: O / l -> bf16 -> global.  The next unit's first PV cannot start before this
    // thread signals its next P, so O is not overwritten while it is being read.
    if (!mbar_wait(&bars->o_done[which], n_units & 1, bars, a.st, 20 + which)) return;
    ++n_units;
    tc_fence_after();
    const int t = u.q_tok + which * kTile + row;
    uint16_t* orow = a.O + u.b * a.osb + u.h * a.osh + (a.seq[u.seq].tok0 + t) * a.ost;
    const float inv = l_run > 0.f ? 1.f / l_run : 0.f;   // a row without any visible key (generic lists only): zeros
#pragma unroll
    for (int q = 0; q < D / 32; ++q) {
      uint32_t ov[32];
      tmem_ld32(tO + q * 32, ov);
      tmem_wait_ld();
      uint32_t w[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] = pack2<kF16>(__uint_as_float(ov[2 * i]) * inv, __uint_as_float(ov[2 * i + 1]) * inv);
      if (t < u.n) {                                 // rows past the end of the sequence (ragged last tile) are dropped
        if (a.o_vec32) {
          // 32-byte stores: every store fills whole 32-byte sectors (a thread owns a row, so the lanes of a
          // store instruction hit 32 different rows; 16-byte stores would touch every sector twice)
          st_global_v8(orow + q * 32, w);
          st_global_v8(orow + q * 32 + 16, w + 8);
        } else {
          uint4* dst = reinterpret_cast<uint4*>(orow + q * 32);
#pragma unroll
          for (int i = 0; i < 4; ++i) dst[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
        }
      }
    }
    if (a.lse != nullptr && t < u.n)
      a.lse[a.seq[u.seq].lse0 + ((long long)u.b * a.Hq + u.h) * u.n + t] = m_run * a.sm_scale + __logf(l_run);
  }
}

// What the tensor cores lose.  QK^T over 64 channels is four accumulations, each rounded towards zero: half a unit in the last place,
// 0.36 x 2^-23 of the running sum on average (the mean of 1/mantissa is 0.72).  The running sums of a large logit grow evenly, so it
// comes out about (1/4 + 1/2 + 3/4 + 1) x 0.36 x 2^-23 = 0.9 x 2^-23 smaller than it is (measured: 1.0 in fp16, 0.7 in bf16, whose
// 16-bit products leave some sums exact).  That cancels in O; lse, where the size of the logits itself counts, gets it back.  A
// tile's P V loses 1 to 3.5 x 2^-23 in the same way (500 to 8000 keys, values of one sign or of both), of which O gets 2 x 2^-23 back.
template <bool kF16> constexpr double kQkLoss = 1.0 + (kF16 ? 1.0 : 0.7) / 8388608.0;
constexpr float kPvLoss = 1.0f + 2.0f / 8388608.0f;

// Heads of 64 channels.  A tile costs a row 128 exponentials as with 128 channels, but half the MMA work and half the output
// columns; that room goes into 32-bit accuracy:
//   * P is stored as the sum of two (fp16) or three (bf16) 16-bit values, each the rounding of what the ones before leave;
//   * each tile's P V starts from zero and is added here, in registers, to nearest (a chain of MMAs over 8192 keys loses up to
//     512 roundings towards zero: 4e-6 of O, against 3e-7 with plain fp32 sums);
//   * changes of the reference maximum, and lse, use the offsets that the exponentials were formed with.
// S is read a half at a time, so that 64 columns of it, their parts of P and the output fit the registers.  Columns of a query
// tile's S region once P is in it, per half (32 columns each): hi of keys 0..63 | lo | hi of keys 64..127 | lo.
// Bound by the instructions of these threads (3700 cycles per pair of tiles in fp16, of which the exponentials need 2050).  Two
// sequences of 6001 tokens, 16 heads, segment 512, block 64, budget 1024: fp16 112 us, bf16 130 us (90 and 88 us with two parts of P
// in either type and one chain of accumulations, whose error was larger than that of plain fp32).
template <bool kF16, int NS>
__device__ __forceinline__ void softmax_role64(const Args<NS>& a, Bars* bars, int which, int warp_in_wg, int lane) {
  constexpr float kShift = kPShift<kF16>;
  const uint32_t tm = bars->tmem_base + (uint32_t(warp_in_wg * 32) << 16);
  const uint32_t tS = tm + which * 128, tO = tm + 256 + which * 64, tX = tm + 384 + which * 64;
  const int row = warp_in_wg * 32 + lane;
  const float c = a.sm_scale * 1.4426950408889634f;   // logits -> log2 units
  uint32_t n_tiles = 0;                               // S tiles consumed so far (all units)
  uint32_t n_units = 0;                               // units finished so far
  float2 o[32];
  auto add = [&](const uint32_t* ov) {                // O += P V of a tile
#pragma unroll
    for (int i = 0; i < 32; ++i) o[i] = __fadd2_rn(o[i], make_float2(__uint_as_float(ov[2 * i]), __uint_as_float(ov[2 * i + 1])));
  };

  for (uint32_t q = 0;; ++q) {
    int x;
    Unit u;
    if (!receive_unit(a, bars, q, lane, &x, &u) || x >= a.n_units || bars->abort_flag) return;
    if (u.cnt == kBadList || u.cnt == kEmptyUnit) continue;
    const int t = u.q_tok + which * kTile + row;
    if (u.cnt == kZeroUnit) {
      write_zero_row<64>(a, u, which, t);
      continue;
    }
    const int my_tiles = which == 0 ? u.nA : u.nB;
    if (my_tiles == 0) continue;                        // this unit has no tile B
    float m_run = -CUDART_INF, l_run = 0.f, offset = 0.f;   // p = 2^(s c + offset), offset = kShift - m_run c rounded
#pragma unroll
    for (int i = 0; i < 32; ++i) o[i] = make_float2(0.f, 0.f);

    for (int jt = 0; jt < my_tiles; ++jt, ++n_tiles) {
      // the QK^T of this tile was issued behind the P V of the one before: both are there
      if (!mbar_wait(&bars->s_full[which], n_tiles & 1, bars, a.st, 10 + which)) return;
      tc_fence_after();

      // last visible offset in each 32 columns of the tile: causal in the own diagonal tile, the listed columns in the last gathered
      // tile, and by token in the tiles of a generic list (128/blk listed blocks, -1 beyond the list)
      bool masked = true;
      int lim[4];
      if (u.generic) {
        const int bpt = kTile / a.blk;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int li = jt * bpt + g * 32 / a.blk;
          lim[g] = li < u.cnt ? t - __ldg(u.list + li) * a.blk - g * 32 % a.blk : -1;
        }
      } else {
        const bool diagonal = jt == my_tiles - 1;
        masked = diagonal || (jt == u.n_past_tiles - 1 && u.last_cols < kTile);
#pragma unroll
        for (int g = 0; g < 4; ++g) lim[g] = (diagonal ? row : u.last_cols - 1) - g * 32;
      }
      auto mask32 = [&](uint32_t* v, int g) {           // columns 32 g to 32 g + 31
        if (masked) {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = i > lim[g] ? 0xff800000u : v[i];
        }
      };
      auto max64 = [&](const uint32_t* v) {
        auto s = [&](int i) { return __uint_as_float(v[i]); };
        float mx0 = s(0), mx1 = s(1), mx2 = s(2), mx3 = s(3);
#pragma unroll
        for (int i = 4; i < 60; i += 8) {
          mx0 = max3(mx0, s(i), s(i + 1)); mx1 = max3(mx1, s(i + 2), s(i + 3));
          mx2 = max3(mx2, s(i + 4), s(i + 5)); mx3 = max3(mx3, s(i + 6), s(i + 7));
        }
        return fmaxf(max3(mx0, s(60), s(61)), max3(max3(mx1, s(62), s(63)), mx2, mx3));
      };
      uint32_t sv[64];                                  // S: keys 0..63, then keys 64..127
      float m_tile;
      {
        uint32_t ov[64], first[64];
        tmem_ld64(tS, first);
        if (jt > 0) {
          tmem_ld64(tO, ov);
          tmem_wait_ld();
          add(ov);
        } else {
          tmem_wait_ld();
        }
        tmem_ld64(tS + 64, sv);
        mask32(first, 0); mask32(first + 32, 1);
        m_tile = max64(first);
      }
      tmem_wait_ld32(sv); tmem_wait_ld32(sv + 32);
      mask32(sv, 2); mask32(sv + 32, 3);
      m_tile = fmaxf(m_tile, max64(sv));
      const float m_new = fmaxf(m_run, m_tile);
      // lazy rescale: keep the old reference maximum while the new one exceeds it by < 2^8
      float f = 1.f;
      if (m_run == -CUDART_INF) {                       // no key seen yet (the first tile; later ones of generic lists only)
        m_run = m_new;
        if (m_new != -CUDART_INF) offset = fmaf(-m_new, c, kShift);
      } else if ((m_new - m_run) * c > kRescaleThreshold) {
        const float offset_new = fmaf(-m_new, c, kShift);
        f = ex2(offset_new - offset);
        m_run = m_new;
        offset = offset_new;
      }
      if (__any_sync(0xffffffffu, f != 1.f)) {
        l_run *= f;
        const float2 f2 = make_float2(f, f);
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = __fmul2_rn(o[i], f2);
      }
      const float2 c2 = make_float2(c, c), off2 = make_float2(offset, offset), minus1 = make_float2(-1.f, -1.f);
      float2 sum2[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) sum2[i] = make_float2(0.f, 0.f);
      auto probabilities = [&](const uint32_t* v, int g) {   // of keys 32 g to 32 g + 31, to tensor memory
        uint32_t hi[16], lo[16], third[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float2 xx = __ffma2_rn(make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), c2, off2);
          float2 p;
          p.x = ex2(xx.x); p.y = ex2(xx.y);
          sum2[i & 3] = __fadd2_rn(sum2[i & 3], p);
          hi[i] = pack2<kF16>(p.x, p.y);
          p = __ffma2_rn(unpack2<kF16>(hi[i]), minus1, p);   // exact: what the part leaves
          lo[i] = pack2<kF16>(p.x, p.y);
          if constexpr (!kF16) {
            p = __ffma2_rn(unpack2<kF16>(lo[i]), minus1, p);
            third[i] = pack2<kF16>(p.x, p.y);
          }
        }
        tmem_st16(tS + (g >> 1) * 64 + (g & 1) * 16, hi);
        tmem_st16(tS + (g >> 1) * 64 + 32 + (g & 1) * 16, lo);
        if constexpr (!kF16) tmem_st16(tX + g * 16, third);
      };
      // the second half of S is at hand; the first comes back 32 columns at a time under the exponentials of the ones before
      probabilities(sv, 2);
      uint32_t sa[32], sb[32];
      tmem_ld32(tS, sa);
      probabilities(sv + 32, 3);
      tmem_wait_ld32(sa);
      mask32(sa, 0);
      tmem_ld32(tS + 32, sb);
      tmem_wait_ld32(sb);                               // before P of keys 0..31 goes over these columns
      probabilities(sa, 0);
      mask32(sb, 1);
      probabilities(sb, 1);
      sum2[0] = __fadd2_rn(__fadd2_rn(sum2[0], sum2[1]), __fadd2_rn(sum2[2], sum2[3]));
      l_run += sum2[0].x + sum2[0].y;
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&bars->p_full[which]);
    }

    // epilogue: the last tile's P V, O / l -> global.  The next unit's first PV cannot start before this thread signals its next P.
    if (!mbar_wait(&bars->o_done[which], n_units & 1, bars, a.st, 20 + which)) return;
    ++n_units;
    tc_fence_after();
    {
      uint32_t ov[64];
      tmem_ld64(tO, ov);
      tmem_wait_ld();
      add(ov);
    }
    uint16_t* orow = a.O + u.b * a.osb + u.h * a.osh + (a.seq[u.seq].tok0 + t) * a.ost;
    const float inv = l_run > 0.f ? kPvLoss / l_run : 0.f;   // a row without any visible key (generic lists only): zeros
    float odd = 0.f;                                     // NaN as soon as one output of the row is NaN or infinite
#pragma unroll
    for (int i = 0; i < 32; ++i) odd = fmaf(o[i].y, 0.f, fmaf(o[i].x, 0.f, odd));
    if (t < u.n) {                                       // rows past the end of the sequence (ragged last tile) are dropped
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = pack2<kF16>(o[q4 * 8 + i].x * inv, o[q4 * 8 + i].y * inv);
        if (a.o_vec32) {
          st_global_v8(orow + q4 * 16, w);               // whole 32-byte sectors (see softmax_role)
        } else {
          uint4* dst = reinterpret_cast<uint4*>(orow + q4 * 16);
          dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
          dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
      }
      if (a.lse != nullptr)
        a.lse[a.seq[u.seq].lse0 + ((long long)u.b * a.Hq + u.h) * u.n + t] =
            float(double(m_run) * (a.sm_scale * kQkLoss<kF16>) + (log(double(l_run)) - 0.693147180559945309417 * (double(m_run) * c + offset)));
    }
    // the warp's rows that came out as NaN or infinite, or saw no key, one after another
    unsigned redo = __ballot_sync(0xffffffffu, !(odd == 0.f && l_run > 0.f && l_run < CUDART_INF_F) && t < u.n);
    for (; redo != 0; redo &= redo - 1) {
      __syncwarp();                                      // the row's own stores come first
      exact_row<kF16>(&a, bars, u.seq, u.b, u.h, u.list, u.cnt, t - lane + (__ffs(redo) - 1), lane);
    }
  }
}

// ---------------------------------------------------------------- producer role
template <int D, int NS>
__device__ __forceinline__ void producer_role(const Args<NS>& a, Bars* bars, uint32_t smem_base, const Maps<NS>& maps, int lane) {
  constexpr int kSlots = Shape<D>::kSlots, kTileBytes = Shape<D>::kTileBytes, kHalves = Shape<D>::kHalves;
  const int bpt = kTile / a.blk;
  uint32_t item = 0;      // K/V tiles issued so far (all units): item i lives in slot i % kSlots
  uint32_t n_units = 0;
  // lane -> box of a gathered tile: block `my_blk` of its 128/blk, half `my_hf` of head_dim
  const int my_blk = lane / kHalves, my_hf = lane % kHalves;
  for (uint32_t q = 0;; ++q) {
    int x;
    Unit u;
    if (!receive_unit(a, bars, q, lane, &x, &u) || x >= a.n_units || bars->abort_flag) return;
    if (lane == 0) mbar_arrive(&bars->taken);
    if (u.cnt == kBadList || u.cnt == kEmptyUnit || u.cnt == kZeroUnit) continue;
    const CUtensorMap* tm = maps.m[NS > 1 ? u.seq : 0];
    // token of this lane's block of gathered tile jt; boxes beyond the list read past the end of the tensor and arrive as zeros
    auto token_of = [&](int jt) {
      const int li = jt * bpt + my_blk;
      return my_blk < bpt && jt < u.n_past_tiles && li < u.n_past ? u.list[li] * a.blk : u.n;
    };
    int tok = token_of(0);
    // Q tiles: the buffer is free once every QK^T of the previous unit has completed
    if (n_units > 0 && !mbar_wait(&bars->q_empty, (n_units - 1) & 1, bars, a.st, 31)) return;
    if (lane == 0) {
      const int nq = u.nB ? 2 : 1;
      mbar_expect_tx(&bars->q_full, nq * kTileBytes);
      for (int w = 0; w < nq; ++w)
        for (int hf = 0; hf < kHalves; ++hf)
          tma_load_4d(smem_base + Shape<D>::kSmemQ + w * kTileBytes + hf * kHalfBytes, tm + kQ, &bars->q_full, hf * 64,
                      u.q_tok + w * kTile, u.h, u.b);
    }
    ++n_units;
    for (int it = 0; it < 2 * u.T; ++it, ++item) {   // 2*jt = K tile jt, 2*jt+1 = V tile jt
      const uint32_t slot = item % kSlots, use = item / kSlots;
      const int jt = it >> 1;
      const bool is_v = it & 1;
      const int next_tok = is_v ? token_of(jt + 1) : 0;   // the next tile's list entries are on their way during the wait
      if (use > 0 && !mbar_wait(&bars->kv_empty[slot], (use - 1) & 1, bars, a.st, 30)) return;
      if (!(a.withhold_v && is_v)) {
        const uint32_t dst = smem_base + Shape<D>::kSmemKV + slot * kTileBytes;
        unsigned long long* bar = &bars->kv_full[slot];
        if (lane == 0) mbar_expect_tx(bar, kTileBytes);
        __syncwarp();
        // one lane per box: the list entries are read and the loads issued side by side, not one after another
        if (jt < u.n_past_tiles) {
          if (my_blk < bpt)
            tma_load_4d(dst + my_hf * kHalfBytes + my_blk * a.blk * 128, tm + (is_v ? kVb : kKb), bar, my_hf * 64, tok, u.kvh, u.b);
        } else if (lane < kHalves) {
          const int ci = jt - u.n_past_tiles;
          const int t0 = ci < u.n_cont ? u.c_tok + ci * kTile : u.d_tok + (ci - u.n_cont) * kTile;
          tma_load_4d(dst + lane * kHalfBytes, tm + (is_v ? kVt : kKt), bar, lane * 64, t0, u.kvh, u.b);
        }
      }
      __syncwarp();
      if (is_v) tok = next_tok;
    }
  }
}

// ---------------------------------------------------------------- MMA role
template <bool kF16, int D>
__device__ __forceinline__ void issue_qk(uint32_t d_tmem, uint32_t q_smem, uint32_t k_smem) {
  const uint64_t base = desc_base(16);
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
    umma_ss(d_tmem, desc_at(base, q_smem + off), desc_at(base, k_smem + off), Idesc<kF16>::qk, kk > 0);
  }
}
template <bool kF16, int D>
__device__ __forceinline__ void issue_pv(uint32_t d_tmem, uint32_t p_tmem, uint32_t x_tmem, uint32_t v_smem, bool acc) {
  const uint64_t base = desc_base(kHalfBytes);   // the two 64-column halves of head_dim are 16 KB apart
  if constexpr (Shape<D>::kSplitP) {
    // the parts of P, smallest first, into a sum that starts from zero (softmax_role64 adds the tiles up)
    if constexpr (!kF16) {
#pragma unroll
      for (int kk = 0; kk < kTile / 16; ++kk)
        umma_ts(d_tmem, x_tmem + kk * 8, desc_at(base, v_smem + kk * 16 * 128), Idesc<kF16, D>::pv, kk > 0);
    }
#pragma unroll
    for (int part = 1; part >= 0; --part)
#pragma unroll
      for (int kk = 0; kk < kTile / 16; ++kk)
        umma_ts(d_tmem, p_tmem + (kk >> 2) * 64 + part * 32 + (kk & 3) * 8, desc_at(base, v_smem + kk * 16 * 128), Idesc<kF16, D>::pv,
                (!kF16 || part == 0 || kk > 0) ? 1u : 0u);
  } else {
#pragma unroll
    for (int kk = 0; kk < kTile / 16; ++kk)
      umma_ts(d_tmem, p_tmem + kk * 8, desc_at(base, v_smem + kk * 16 * 128), Idesc<kF16, D>::pv, (acc || kk > 0) ? 1u : 0u);
  }
}

template <bool kF16, int D, int NS>
__device__ __forceinline__ void mma_role(const Args<NS>& a, Bars* bars, uint32_t smem_base, int lane) {
  constexpr int kSlots = Shape<D>::kSlots, kTileBytes = Shape<D>::kTileBytes;
  const uint32_t tm = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  const uint32_t tS[2] = {tm, tm + 128}, tO[2] = {tm + 256, tm + 256 + D}, tX[2] = {tm + 384, tm + 448};   // tX: 64 channels only
  const uint32_t qA = smem_base + Shape<D>::kSmemQ, qB = qA + kTileBytes;
  uint32_t item0 = 0;                 // first K/V item of the current unit
  uint32_t nA = 0, nB = 0;            // P tiles consumed so far per query tile (all units)
  uint32_t n_units = 0;
  auto slot_addr = [&](uint32_t item) { return smem_base + Shape<D>::kSmemKV + (item % kSlots) * kTileBytes; };
  auto full_wait = [&](uint32_t item) {
    return mbar_wait(&bars->kv_full[item % kSlots], (item / kSlots) & 1, bars, a.st, 40);
  };
  for (uint32_t q = 0;; ++q) {
    int x;
    Unit u;
    if (!receive_unit(a, bars, q, lane, &x, &u) || x >= a.n_units || bars->abort_flag) return;
    if (u.cnt == kBadList || u.cnt == kEmptyUnit || u.cnt == kZeroUnit) continue;
    const int T = u.T, TA = u.nA;
    const bool hasB = u.nB > 0;
    if (!mbar_wait(&bars->q_full, n_units & 1, bars, a.st, 41)) return;
    if (!full_wait(item0)) return;
    tc_fence_after();
    issue_qk<kF16, D>(tS[0], qA, slot_addr(item0)); umma_commit(&bars->s_full[0]);
    if (hasB) { issue_qk<kF16, D>(tS[1], qB, slot_addr(item0)); umma_commit(&bars->s_full[1]); }
    umma_commit(&bars->kv_empty[item0 % kSlots]);
    if (T == 1) umma_commit(&bars->q_empty);               // a one-tile unit has no further QK^T
    for (int jt = 0; jt < T; ++jt) {
      const bool has_next = jt + 1 < T;
      const uint32_t iv = item0 + 2 * jt + 1, ik = item0 + 2 * (jt + 1);
      if (has_next && !full_wait(ik)) return;
      if (!full_wait(iv)) return;
      const uint32_t v_smem = slot_addr(iv), kn_smem = slot_addr(ik);
      if (jt < TA) {
        if (!mbar_wait(&bars->p_full[0], nA & 1, bars, a.st, 42)) return;
        ++nA;
        tc_fence_after();
        issue_pv<kF16, D>(tO[0], tS[0], tX[0], v_smem, jt > 0);
        if (jt + 1 < TA) { issue_qk<kF16, D>(tS[0], qA, kn_smem); umma_commit(&bars->s_full[0]); }
        else umma_commit(&bars->o_done[0]);
      }
      if (hasB) {
        if (!mbar_wait(&bars->p_full[1], nB & 1, bars, a.st, 43)) return;
        ++nB;
        tc_fence_after();
        issue_pv<kF16, D>(tO[1], tS[1], tX[1], v_smem, jt > 0);
      }
      umma_commit(&bars->kv_empty[iv % kSlots]);             // every PV that reads this V tile has been issued
      if (has_next) {
        if (hasB) { issue_qk<kF16, D>(tS[1], qB, kn_smem); umma_commit(&bars->s_full[1]); }
        umma_commit(&bars->kv_empty[ik % kSlots]);
        if (jt + 1 == T - 1) umma_commit(&bars->q_empty);   // that was the unit's last QK^T: Q may be replaced
      } else if (hasB) {
        umma_commit(&bars->o_done[1]);
      }
    }
    item0 += 2 * T;
    ++n_units;
  }
}

// ---------------------------------------------------------------- kernel
template <bool kF16, int D, int NS>
__global__ void __launch_bounds__(kThreads, 1)
attention_sm100_kernel(const __grid_constant__ Maps<NS> maps, const __grid_constant__ Args<NS> a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t smem_base = (raw + 1023u) & ~1023u;
  static_assert(sizeof(Bars) <= kBarBytes, "barrier block too small");
  Bars* bars = reinterpret_cast<Bars*>(smem_raw + (smem_base - raw) + Shape<D>::kSmemBar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->q_empty, 1);
    for (int i = 0; i < Shape<D>::kSlots; ++i) { mbar_init(&bars->kv_full[i], 1); mbar_init(&bars->kv_empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->s_full[i], 1); mbar_init(&bars->p_full[i], 128); mbar_init(&bars->o_done[i], 1); }
    mbar_init(&bars->clc_full, 1);
    mbar_init(&bars->taken, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&bars->sched_full[i], 1); mbar_init(&bars->sched_empty[i], 10); }   // 8 softmax warps, producer, MMA
    bars->abort_flag = 0;
    bars->beat = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 8 && lane < kMaps && NS == 1) prefetch_tmap(&maps.m[0][lane]);
  if (warp == 9) { tmem_alloc(&bars->tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();

  // Register re-partition.  The pool is what the CTA was launched with (384 threads x 168):
  // 256 x 216 + 128 x 64 = 63488 fits; asking for more than the pool would block forever.
  static_assert(kRegPoolNeeded <= kThreads * 168, "setmaxnreg budget exceeds the launch allocation");
  if (warp < 8) {
    reg_inc<216>();
    if constexpr (D == 64) softmax_role64<kF16, NS>(a, bars, warp >> 2, warp & 3, lane);
    else softmax_role<kF16, NS>(a, bars, warp >> 2, warp & 3, lane);
  } else {
    reg_dec<64>();
    if (warp == 8) producer_role<D, NS>(a, bars, smem_base, maps, lane);
    else if (warp == 9) mma_role<kF16, D, NS>(a, bars, smem_base, lane);
    else if (warp == 10) scheduler_role<NS>(a, bars, lane);
  }
  if (bars->abort_flag) {
    // give copies and MMAs still in flight time to land before the CTA's resources go away
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(bars->tmem_base, 512);
}

// ---------------------------------------------------------------- host side
// [B, H, n, d] 16-bit with element strides (sb, sh, st); box = 64 columns x `rows` tokens
bool make_map(CUtensorMap* map, const void* base, int B, int H, int n, int d, const int64_t* s, int rows, bool f16) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[4] = {cuuint64_t(d), cuuint64_t(n), cuuint64_t(H), cuuint64_t(B)};
  // nothing reads the stride of a dimension of extent 1, and the encoder takes no stride of 2^40 bytes
  auto stride = [&](int extent, int64_t x) { return extent > 1 ? cuuint64_t(x) * 2 : cuuint64_t(d) * 2; };
  cuuint64_t strides[3] = {stride(n, s[2]), stride(H, s[1]), stride(B, s[0])};
  cuuint32_t box[4] = {64, cuuint32_t(rows), 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool sm100_path_applies(const cp_params& p, const Dims& m) {
  return (p.dtype == CP_BF16 || p.dtype == CP_F16) && (m.d == 128 || m.d == 64) && m.seg % kTile == 0 && (m.blk == 32 || m.blk == 64 || m.blk == 128) &&
         !(p.flags & CP_FLAG_FORCE_SIMT);
}

namespace {

template <bool kF16, int D, int NS>
int launch_variant(const Maps<NS>& maps, const Args<NS>& a, cudaStream_t s) {
  auto kern = attention_sm100_kernel<kF16, D, NS>;
  // setmaxnreg.inc blocks forever when the CTA's register pool (threads x registers the kernel was compiled
  // to) is smaller than what the roles ask for, and no bounded wait covers that: check the real allocation of
  // this build once per variant and refuse to launch instead.
  static int regs_ok = 0;   // 0 = not checked yet, 1 = fits, -1 = does not fit
  if (regs_ok == 0) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return CP_ERR_CUDA;
    regs_ok = (fa.numRegs * kThreads >= kRegPoolNeeded) ? 1 : -1;
  }
  if (regs_ok < 0) return CP_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<D>::kSmemTotal) != cudaSuccess)
    return CP_ERR_CUDA;
  return launch_pdl(kern, dim3(unsigned(a.n_units)), kThreads, Shape<D>::kSmemTotal, s, maps, a);
}

// pairs of 128-row query tiles in a segment: a segment can be longer than every sequence, and empty units cost a hand-over each
int pairs_per_segment(int seg, const SeqSlot* slots, int n_seqs) {
  int rows = 0;
  for (int i = 0; i < n_seqs; ++i) rows = std::max(rows, std::min(seg, slots[i].len));
  return ((rows + kTile - 1) / kTile + 1) / 2;
}

// units of a launch that have query rows
long long count_units(const Dims& m, const SeqSlot* slots, int n_seqs, bool dense) {
  auto pairs = [](int rows) { return (rows + 2 * kTile - 1) / (2 * kTile); };
  long long per_head = 0;
  for (int i = 0; i < n_seqs; ++i)
    per_head += dense ? pairs(slots[i].len) : (long long)(slots[i].len / m.seg) * pairs(m.seg) + pairs(slots[i].len % m.seg);
  return per_head * m.B * m.Hq;
}

// Whether pairs of CTAs take a launch in less time than single ones.  Units are handed out one ahead, so the SMs go through them in
// rounds, as it were, longest units first, and each round lasts as long as its longest unit: rounds of 148 units on single CTAs, of 74 on
// pairs, which take 0.5 of a single CTA's time per tile of a short unit, 0.62 of a long one (0.60 without a list), and 0.75 tiles more per launch.
// Over 336 launches (37 to 3000 units of 2 to 1200 tiles; 1 / 1, 8 / 2 and 32 / 8 heads; loops of 0.1 s) the choice costs 0.4 % on average against
// the faster kernel; the worst seen, single CTAs / pairs, us: 8 / 2 heads, 7104 tokens, budget 8192, 113 / 123, on pairs; 16 / 4 heads, 4000 tokens,
// budget 8192, 90 / 81, on single ones.
// Single CTAs / pairs, us: segment 512, budget 1024: 37 units 22.5 / 15.8, 111 23.3 / 23.0, 222 36.8 / 31.5, 296 39.5 / 41.5; segment 1024, budget
// 4096: 74 64.3 / 44.2, 110 64.6 / 73.6, 185 112 / 105, 260 128 / 144, 444 206 / 231; dense, 8 / 2 heads: 80 units 39.1 / 30.3, 192 105 / 92, 296 201 /
// 204, 448 395 / 445.
// With more than three units per SM the ends of the rounds no longer count.  Long units then cost pairs 5 to 15 % more (power); short ones cost
// the same in long loops and 4 to 20 % less between other kernels, as their beginnings and ends overlap: whole layer of 8192 tokens (1024
// units) 163.7 / 161.5 us; units of two tiles 12 % more (segment = budget = 256, 2072 units 107 / 122), of four 0.5 % less, so the line lies at 3.5
// on average.  Beyond 14 per SM not even the former (whole layers, a batch of 3296 units 474 / 484).
bool pairs_are_faster(const Dims& m, const SeqSlot* slots, int n_seqs, bool dense, bool long_units) {
  constexpr int kMany = 3 * 148;
  const long long units = count_units(m, slots, n_seqs, dense);
  if (units > kMany) return !long_units && units <= 14 * 148 && 2 * ((m.k - m.r) * (long long)m.blk + m.seg / 2 + kTile) >= 7 * kTile;
  int tiles[kMany], classes = 0;                    // of each unit of a head
  for (int i = 0; i < n_seqs; ++i) {
    const int seg = dense ? slots[i].len : m.seg;
    for (int j = 0; j * seg < slots[i].len; ++j) {
      const int rows = std::min(seg, slots[i].len - j * seg);
      const long long past = dense ? 0 : std::min((long long)j * m.r, (long long)m.k - m.r) * m.blk;
      for (int x = 0; x < rows; x += 2 * kTile)
        tiles[classes++] = int((past + kTile - 1) / kTile) + x / kTile + (x + kTile < rows ? 2 : 1);
    }
  }
  std::sort(tiles, tiles + classes, [](int a, int b) { return a > b; });
  const long long heads = (long long)m.B * m.Hq;
  auto rounds = [&](int places) {
    long long sum = 0;
    for (long long x = 0; x < units; x += places) sum += tiles[x / heads];
    return sum;
  };
  const long long single = rounds(148), pair = rounds(74);
  return long_units ? (dense ? 60 : 62) * pair + 75 < 100 * single : 50 * pair + 75 < 100 * single;
}

// (segment, pair)s that have query rows, by the tiles they stream, longest first (counting sort; equal ones from the last
// segment down).  Returns their number, 0 when there are more than the table holds.
template <int NS>
int order_units(Args<NS>& a) {
  const int pp = a.pp;
  if ((long long)a.n_segs * pp > kMaxOrder) return 0;
  constexpr int kCosts = 256;
  uint16_t cost[kMaxOrder];
  int start[kCosts + 1] = {0};
  const int m = a.k - a.r;                          // blocks before the segment that a list can hold
  int total = 0;
  for (int i = 0; i < a.n_seqs; ++i)
    for (int j = 0; j < a.seq[i].n1; ++j)
      for (int p = 0; p < pp; ++p) {
        const long long past = (long long)j * a.r < m ? (long long)j * a.r : m;
        const long long c = j * a.seg + p * 256 < a.seq[i].n ? (past * a.blk + kTile - 1) / kTile + 2 * p + 2 : 0;
        const int cc = int(c < kCosts ? c : kCosts - 1);
        cost[(a.seq[i].seg0 + j) * pp + p] = uint16_t(cc);
        if (cc > 0) { ++start[kCosts - cc]; ++total; }   // start[x]: units of the costs above x's
      }
  for (int c = 1; c <= kCosts; ++c) start[c] += start[c - 1];
  for (int e = a.n_segs * pp - 1; e >= 0; --e)
    if (cost[e] > 0) a.order[start[kCosts - cost[e] - 1]++] = uint16_t(e);
  return total;
}

// slots[0..n_seqs): the sequences of one launch (a single problem is one sequence that starts at 0)
template <int NS>
int launch_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, int n_seqs, const void* Q, const void* K, const void* V,
                const int32_t* idx, const int32_t* cnt, void* O, float* lse, DeviceStatus* st, bool dense, cudaStream_t s) {
  const bool f16 = p.dtype == CP_F16;
  Maps<NS> maps;
  OMaps<NS> o_maps;
  Args<NS> a;
  // Moving every kEmulEvery-th pair of exponentials from the MUFU to the FMA pipes pays where units are long and the
  // kernel sits at the power cap (measured in 60-step loops: 1.6 % at 32 K/V tiles per unit) and costs where units are
  // short (3 % at 8 tiles per unit, the paper's operating point); a unit streams at most k*blk/128 tiles.
  a.emul = (dense || (long long)m.k * m.blk >= 12 * kTile) ? 1 : 0;
  // The kernel of CTA pairs (attention_pair_sm100.cu) takes heads of 128 channels whose units have two query tiles (segments of an odd number
  // of tiles would leave half of every pair idle), where it is the faster one.  The results are the same bits.
  const bool pair = m.d == 128 && (dense || m.seg % (2 * kTile) == 0) && pairs_are_faster(m, slots, n_seqs, dense, a.emul != 0);
  a.n_segs = 0;
  a.pp = pairs_per_segment(m.seg, slots, n_seqs);
  long long kv_tokens = 0;
  for (int i = 0; i < n_seqs; ++i) {
    const SeqSlot& q = slots[i];
    auto at = [&](const void* base, const int64_t* stride) { return static_cast<const char*>(base) + q.tok * stride[2] * m.es; };
    CUtensorMap* t = maps.m[i];
    if (!make_map(t + kQ, at(Q, p.q_stride), m.B, m.Hq, q.len, m.d, p.q_stride, kTile, f16) ||
        !make_map(t + kKb, at(K, p.k_stride), m.B, m.Hkv, q.len, m.d, p.k_stride, pair ? std::min(m.blk, 64) : m.blk, f16) ||
        !make_map(t + kVb, at(V, p.v_stride), m.B, m.Hkv, q.len, m.d, p.v_stride, m.blk, f16) ||
        !make_map(t + kKt, at(K, p.k_stride), m.B, m.Hkv, q.len, m.d, p.k_stride, pair ? 64 : kTile, f16) ||
        !make_map(t + kVt, at(V, p.v_stride), m.B, m.Hkv, q.len, m.d, p.v_stride, kTile, f16) ||
        (pair && !make_map(&o_maps.m[i], at(O, p.o_stride), m.B, m.Hq, q.len, m.d, p.o_stride, 32, f16)))
      return CP_ERR_CUDA;
    Seq& x = a.seq[i];
    x.n = q.len; x.n1 = (q.len + m.seg - 1) / m.seg; x.n2 = (q.len + m.blk - 1) / m.blk;
    x.seg0 = a.n_segs;
    x.tok0 = q.tok; x.idx0 = q.idx; x.cnt0 = q.cnt; x.lse0 = int64_t(m.Hq) * q.tok;
    a.n_segs += x.n1;
    kv_tokens += q.len;
  }
  a.n_seqs = n_seqs;
  a.idx = idx; a.cnt = cnt; a.O = static_cast<uint16_t*>(O); a.lse = lse; a.st = st;
  a.B = m.B; a.Hq = m.Hq; a.Hkv = m.Hkv; a.g = m.g; a.seg = m.seg; a.blk = m.blk; a.k = m.k;
  a.r = m.r;
  a.osb = p.o_stride[0]; a.osh = p.o_stride[1]; a.ost = p.o_stride[2];
  a.Q = static_cast<const uint16_t*>(Q); a.K = static_cast<const uint16_t*>(K); a.V = static_cast<const uint16_t*>(V);
  for (int i = 0; i < 3; ++i) { a.qs[i] = p.q_stride[i]; a.ks[i] = p.k_stride[i]; a.vs[i] = p.v_stride[i]; }
  a.sm_scale = p.sm_scale; a.dense = dense ? 1 : 0;
  // a unit is two 128-row query tiles (one when a segment, or the sequence, has an odd tile count)
  const long long units = dense ? (long long)m.B * m.Hq * (((m.n + kTile - 1) / kTile + 1) / 2)
                                : (long long)m.B * m.Hq * a.n_segs * a.pp;
  if (units > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  a.n_units = int(units);
  // K and V of every head up to 160 MB (measured on both sides: see decode_unit; the L2 has 126 MB); a batch of sequences always: over
  // lists the order pays at every size measured there, and one launch saves the end of another (two prompts of 131072 tokens,
  // segment 1024, budget 4096, whole layers: 15.8 ms in one batch, 16.1 ms in two calls; of 65536 7.6 / 7.8 ms)
  a.long_first = (NS > 1 || kv_tokens * m.B * m.Hkv * m.d * m.es * 2 <= 160ll << 20) ? 1 : 0;
  if (a.long_first && !dense) {
    const int entries = order_units(a);
    if (entries > 0) a.n_units = m.B * m.Hq * entries;
    else a.long_first = 0;                          // more segments than the table holds (never for a batch: see below)
  }
  a.withhold_v = (p.flags & CP_FLAG_TEST_WITHHOLD_V) ? 1 : 0;
  a.o_vec32 = (reinterpret_cast<uintptr_t>(O) % 32 == 0 && p.o_stride[0] % 16 == 0 && p.o_stride[1] % 16 == 0 && p.o_stride[2] % 16 == 0) ? 1 : 0;
  if (pair) return launch_attention_pair<NS>(maps, o_maps, a, f16, s);
  if (m.d == 64) return f16 ? launch_variant<true, 64, NS>(maps, a, s) : launch_variant<false, 64, NS>(maps, a, s);
  return f16 ? launch_variant<true, 128, NS>(maps, a, s) : launch_variant<false, 128, NS>(maps, a, s);
}

}  // namespace

int launch_attention_sm100(const cp_params& p, const Dims& m, const void* Q, const void* K, const void* V,
                           const int32_t* idx, const int32_t* cnt, void* O, float* lse, DeviceStatus* st,
                           bool dense, cudaStream_t s) {
  const SeqSlot one{0, 0, 0, 0, m.n};
  return launch_seqs<1>(p, m, &one, 1, Q, K, V, idx, cnt, O, lse, st, dense, s);
}

int launch_attention_sm100_varlen(const cp_params& p, const Dims& m, const SeqSlot* slots, int n_seqs, const void* Q, const void* K,
                                  const void* V, const int32_t* idx, const int32_t* cnt, void* O, float* lse, DeviceStatus* st,
                                  cudaStream_t s) {
  for (int i = 0; i < n_seqs;) {
    // as many sequences as a launch has tensor maps and unit entries for; a lone one takes the single-problem launch
    int c = 0;
    long long segs = 0;
    while (c < kMaxSeqs && i + c < n_seqs) {
      segs += (slots[i + c].len + m.seg - 1) / m.seg;
      if (segs * pairs_per_segment(m.seg, slots + i, c + 1) > kMaxOrder) break;
      ++c;
    }
    const int rc = c > 1 ? launch_seqs<kMaxSeqs>(p, m, slots + i, c, Q, K, V, idx, cnt, O, lse, st, false, s)
                         : launch_seqs<1>(p, m, slots + i, 1, Q, K, V, idx, cnt, O, lse, st, false, s);
    if (rc != CP_OK) return rc;
    i += c > 1 ? c : 1;
  }
  return CP_OK;
}

}  // namespace cp
