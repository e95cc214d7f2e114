// K3: critical block selection (Algorithm 2, line 8).  One CTA per (batch, query head,
// segment j).  The r diagonal blocks are always taken; the other m = k - r slots go to the
// strictly-past blocks with the largest score, ties to the larger block index.  Exact: order-preserving
// 64-bit keys are held in registers; a histogram over one 8-bit digit after the other leaves the blocks
// that may hold the m-th largest score, until they are few enough to be ranked against each other (usually
// after the first digit), and an ordered compaction by warp ballots writes the list ascending.
#include "cp_common.cuh"

namespace cp {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ unsigned long long ordered_key(double x) {
  if (x == 0.0) x = 0.0;   // -0.0 and +0.0 compare equal and must map to one key
  unsigned long long u = (unsigned long long)__double_as_longlong(x);
  return (u & 0x8000000000000000ull) ? ~u : (u | 0x8000000000000000ull);
}

constexpr int kRank = 32;        // as many candidates are ranked against each other instead of by a further digit
constexpr int kLastLevel = 9;

// The digit of a level of the search; larger keys (equal keys: larger indices) never have the smaller digit.
//   0     sign, exponent and four bits of the mantissa, clamped to scores from -2^12 to -2^-4: ln S lies there, so that this
//         digit alone spreads a row over 256 bins (its plain top byte is the same for nearly all of them)
//   1-8   the bytes of the key
//   9     the block index (all keys left are equal)
__device__ __forceinline__ int digit_of(int level, unsigned long long key, int b) {
  const uint32_t hi = uint32_t(key >> 32);
  if (level == 0) return min(max(int(hi >> 16) - 0x3F50, 0), 255);
  if (level == kLastLevel) return b >> 5;
  return ((level <= 4 ? hi : uint32_t(key)) >> ((32 - 8 * level) & 31)) & 0xff;
}

// KPT = keys per thread at most.  The past blocks are dealt to the warps in consecutive parts of equal size, whatever the segment,
// and inside a part lane by lane, so that reads and the written list are coalesced and the list is in order.  The kernel is bound by
// latency: barriers, shared-memory atomics, one read of a row of scores.  When a thread owned KPT consecutive blocks each load of a
// warp touched 32 lines, and the first two of three to four byte digits hit one or two bins.  Before / now, us, calls back to back in a
// graph, 32 heads, segment 512, block 32: 1300 tokens 4.3 / 2.5, 4096 4.9 / 4.2, 8192 5.6 / 5.1, 16384 8.8 / 7.2, 131072 142 / 120;
// segment 1024, block 128, 131072 tokens 26.9 / 23.0.  Candidates ranked, 32 / 64 / 128: 8192 tokens 5.1 / 5.3 / 6.8; several lanes
// per candidate 8.4.
// `pool` > 1: one CTA per (batch, KV head, segment); the key of a block is the largest of the pool's `pool`
// consecutive query heads' scores, and the one list is written for each of them.  n_sink / n_local: the first
// n_sink blocks and the n_local blocks right before the segment get the largest possible key, so they are taken
// before any scored block (the host has checked that they fit into the k - r free slots).
// Resident CTAs per SM are set by registers; 16 keys per thread are held to 64 registers (4 CTAs).
// One sequence of the launch (a single problem is one).
struct SelectSeq { const double* S; int32_t *idx, *cnt; int n1, n2, cta_begin; };
template <int NS> struct SelectArgs { SelectSeq s[NS]; int n; };

template <int KPT, int NS>
__global__ void __launch_bounds__(kThreads, KPT <= 4 ? 5 : (KPT <= 16 ? 4 : 2))
select_kernel(const __grid_constant__ SelectArgs<NS> a, int r, int k, int pool, int n_sink, int n_local, int past_fixed) {
  __shared__ unsigned int hist[256];
  __shared__ int warp_sum[kWarps];
  __shared__ int bin_sh, remaining_sh, count_sh, n_cand;
  __shared__ unsigned long long cand_key[kRank], thr_sh;
  __shared__ int cand_blk[kRank], thr_blk_sh;
  int si = 0;
  while (NS > 1 && si + 1 < a.n && int(blockIdx.x) >= a.s[si + 1].cta_begin) ++si;
  const SelectSeq& sq = a.s[NS > 1 ? si : 0];
  const double* S = sq.S;
  int32_t *idx = sq.idx, *cnt = sq.cnt;
  const int n1 = sq.n1, n2 = sq.n2, cta = int(blockIdx.x) - sq.cta_begin;
  pdl_trigger();
  pdl_wait(S);

  // CTA -> (batch * heads / pool + pooled head, segment); its first query head's unit is `unit`
  const int j = cta % n1;
  const int unit = (cta / n1) * pool * n1 + j;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* row = S + size_t(unit) * n2;
  const int past = past_fixed >= 0 ? past_fixed : j * r;   // past_fixed: the caller names the first diagonal block (decoding: the last block)
  const int rj = min(n2, past + r) - past;   // diagonal blocks of this segment (fewer in a short last segment)
  const int m = k - rj;

  if (past <= m) {
    // every visible block fits in the budget
    const int c = past + rj;
    for (int u = 0; u < pool; ++u) {
      int32_t* out = idx + (size_t(unit) + size_t(u) * n1) * k;
      for (int i = tid; i < k; i += kThreads) out[i] = i < c ? i : -1;
      if (tid == 0) cnt[unit + u * n1] = c;
    }
    return;
  }

  if (m == 0) {
    // the budget holds the diagonal blocks only
    for (int u = 0; u < pool; ++u) {
      int32_t* out = idx + (size_t(unit) + size_t(u) * n1) * k;
      for (int i = tid; i < k; i += kThreads) out[i] = i < rj ? past + i : -1;
      if (tid == 0) cnt[unit + u * n1] = rj;
    }
    return;
  }

  const int part = (past + kThreads - 1) / kThreads * 32;   // blocks per warp, a multiple of 32, at most 32 * KPT
  const int b0 = warp * part + lane, b_end = min(past, (warp + 1) * part);
  unsigned long long key[KPT];
  unsigned alive = 0;                        // bit s: block b0 + 32 s may be the one that holds the m-th largest key
#pragma unroll
  for (int s = 0; s < KPT; ++s) {
    key[s] = 0ull;
    if (b0 + 32 * s < b_end) alive |= 1u << s;
  }
#pragma unroll 1
  for (int u = 0; u < pool; ++u, row += size_t(n1) * n2) {
#pragma unroll
    for (int s = 0; s < KPT; ++s)
      if (alive >> s & 1u) key[s] = max(key[s], ordered_key(__ldg(row + b0 + 32 * s)));
  }
  if ((n_sink | n_local) != 0) {             // forced blocks
#pragma unroll
    for (int s = 0; s < KPT; ++s)
      if (b0 + 32 * s < n_sink || b0 + 32 * s >= past - n_local) key[s] = ~0ull;
  }
  hist[tid] = 0;
  if (tid == 0) n_cand = 0;
  __syncthreads();

  // ---- the block that holds the m-th largest past score (equal scores: the larger index is the larger) ----
  int remaining = m;                         // its rank among those alive
  int count = past;                          // how many are alive
  unsigned above_mask = 0;                   // bit s: the block is certainly taken
  for (int level = 0; count > kRank && level <= kLastLevel;) {
#pragma unroll
    for (int s = 0; s < KPT; ++s)
      if (alive >> s & 1u) atomicAdd(&hist[digit_of(level, key[s], b0 + 32 * s)], 1u);
    __syncthreads();
    // suffix sums over the 256 bins: thread t owns bin t; above(t) = keys with a larger digit
    const int mine = int(hist[tid]);
    hist[tid] = 0;                 // only its owner reads a bin, so it can be cleared for the next level right away
    int incl = mine;               // inclusive suffix sum within the warp (towards higher lanes)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_down_sync(0xffffffffu, incl, o);
      if (lane + o < 32) incl += v;
    }
    if (lane == 0) warp_sum[warp] = incl;
    __syncthreads();
    int above = incl - mine;
    for (int w = warp + 1; w < kWarps; ++w) above += warp_sum[w];
    if (above < remaining && remaining <= above + mine) {   // exactly one bin satisfies this
      bin_sh = tid;
      remaining_sh = remaining - above;
      count_sh = mine;
    }
    __syncthreads();
    const int bin = bin_sh;
    remaining = remaining_sh;
    count = count_sh;
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
      if (!(alive >> s & 1u)) continue;
      const int dg = digit_of(level, key[s], b0 + 32 * s);
      if (dg > bin) above_mask |= 1u << s;
      if (dg != bin) alive &= ~(1u << s);
    }
    level = level == 0 && bin > 0 && bin < 255 ? 3 : level + 1;   // not clamped: the keys left agree in their top two bytes
  }
  // at most kRank blocks are left (the index digit leaves 32): each counts those before it
#pragma unroll
  for (int s = 0; s < KPT; ++s)
    if (alive >> s & 1u) {
      const int at = atomicAdd(&n_cand, 1);
      cand_key[at] = key[s];
      cand_blk[at] = b0 + 32 * s;
    }
  __syncthreads();
  if (tid < count) {
    const unsigned long long kk = cand_key[tid];
    const int bb = cand_blk[tid];
    int before = 0;
    for (int i = 0; i < count; ++i) before += (cand_key[i] > kk) | ((cand_key[i] == kk) & (cand_blk[i] > bb));
    if (before == remaining - 1) { thr_sh = kk; thr_blk_sh = bb; }
  }
  __syncthreads();
  const unsigned long long thr = thr_sh;
  const int thr_blk = thr_blk_sh;
  unsigned take = above_mask;
#pragma unroll
  for (int s = 0; s < KPT; ++s)
    if ((alive >> s & 1u) && (key[s] > thr || (key[s] == thr && b0 + 32 * s >= thr_blk))) take |= 1u << s;

  // ---- ordered compaction ----
  int n_warp = 0;
#pragma unroll
  for (int s = 0; s < KPT; ++s) n_warp += __popc(__ballot_sync(0xffffffffu, take >> s & 1u));
  if (lane == 0) warp_sum[warp] = n_warp;
  __syncthreads();
  int first = 0;
  for (int w = 0; w < warp; ++w) first += warp_sum[w];
  for (int u = 0; u < pool; ++u) {           // the same list for every head of the pool
    int32_t* out = idx + (size_t(unit) + size_t(u) * n1) * k;
    int pos = first;
#pragma unroll
    for (int s = 0; s < KPT; ++s) {
      const unsigned taken = __ballot_sync(0xffffffffu, take >> s & 1u);
      const int at = pos + __popc(taken & ((1u << lane) - 1u));
      if ((take >> s & 1u) && at < m) out[at] = b0 + 32 * s;
      pos += __popc(taken);
    }
    for (int i = tid; i < rj; i += kThreads) out[m + i] = past + i;   // diagonal blocks
    if (tid == 0) cnt[unit + u * n1] = k;
  }
}

template <int NS>
int launch_args(const cp_params& p, const Dims& m, const SelectArgs<NS>& a, long long units, int n2_max, int past_fixed, cudaStream_t st) {
  const int pool = (p.flags & CP_FLAG_SHARED_GROUP_LISTS) ? m.g : 1;
  const int n_sink = p.forced_blocks & 0xffff, n_local = (p.forced_blocks >> 16) & 0xffff;
  if (units > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  const int kpt = (n2_max + kThreads - 1) / kThreads;
  const dim3 grid(static_cast<unsigned>(units));
  if (kpt <= 4) return launch_pdl(select_kernel<4, NS>, grid, kThreads, 0, st, a, m.r, m.k, pool, n_sink, n_local, past_fixed);
  if (kpt <= 8) return launch_pdl(select_kernel<8, NS>, grid, kThreads, 0, st, a, m.r, m.k, pool, n_sink, n_local, past_fixed);
  if (kpt <= 16) return launch_pdl(select_kernel<16, NS>, grid, kThreads, 0, st, a, m.r, m.k, pool, n_sink, n_local, past_fixed);
  if (kpt <= 32) return launch_pdl(select_kernel<32, NS>, grid, kThreads, 0, st, a, m.r, m.k, pool, n_sink, n_local, past_fixed);
  return CP_ERR_UNSUPPORTED;
}

}  // namespace

int launch_select(const cp_params& p, const Dims& m, const double* S, int32_t* idx, int32_t* cnt,
                  cudaStream_t st, int past_fixed) {
  SelectArgs<1> a;
  a.s[0] = {S, idx, cnt, m.n1, m.n2, 0};
  a.n = 1;
  const int pool = (p.flags & CP_FLAG_SHARED_GROUP_LISTS) ? m.g : 1;
  return launch_args<1>(p, m, a, (long long)m.B * (m.Hq / pool) * m.n1, m.n2, past_fixed, st);
}

int launch_select_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, int n_seqs, const double* S, int32_t* idx, int32_t* cnt,
                       cudaStream_t st) {
  const int pool = (p.flags & CP_FLAG_SHARED_GROUP_LISTS) ? m.g : 1;
  for (int i = 0; i < n_seqs; i += kSeqsPerLaunch) {
    SelectArgs<kSeqsPerLaunch> a;
    a.n = 0;
    long long units = 0;
    int n2_max = 0;
    for (int x = i; x < n_seqs && x < i + kSeqsPerLaunch; ++x) {
      const Dims q = seq_dims(m, slots[x].len);
      if (units > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
      a.s[a.n++] = {S + slots[x].s, idx + slots[x].idx, cnt + slots[x].cnt, q.n1, q.n2, int(units)};
      units += (long long)(m.Hq / pool) * q.n1;
      if (q.n2 > n2_max) n2_max = q.n2;
    }
    const int rc = launch_args<kSeqsPerLaunch>(p, m, a, units, n2_max, -1, st);
    if (rc != CP_OK) return rc;
  }
  return CP_OK;
}

}  // namespace cp
