// K2: criticality scores from the representatives (Algorithm 1, lines 9-14), in fp64 and in
// the log domain.  One CTA handles one segment j for U query heads of the same KV group: the
// key summaries of the group are read and widened to fp64 once and used for all U heads.
// Per head it forms the four logit rows l1..l4 against every key block, their log-sum-exps, and
//   ln S = max( ln((S1+S3)/2), ln((S2+S4)/2) ),  mask,  ln(alpha S + (1-alpha) S').
// The representatives are exact in the input dtype and every product is exact in fp64, so this differs
// from an fp64 CPU evaluation only by summation order, libm rounding and the 1e-15 of the ln(1 + e^-x) table.
#include <cooperative_groups.h>
#include <math_constants.h>

#include "score_common.cuh"

namespace cp {
namespace {

// Threads per CTA.  A CTA's phases (products on the fp64 tensor cores, log-sum-exps, combination) use different units one after
// another; with 256 threads two CTAs share an SM and work in different phases (the registers of 512 allow one).  With no more CTAs than
// SMs a CTA has its SM to itself anyway and is faster with 512.
// One CTA of 512 threads / two of 256 per SM, us, in graphs, 32 / 8 heads, segment 512: 16384 tokens, block 32 (256 CTAs) 35.9 / 33.6, block 64 23.4 /
// 19.4; 32768 tokens, block 64, fused (512 CTAs) 77.0 / 70.0.
constexpr int kThreadsFew = 512, kThreadsMany = 256;

// Shared memory: logits lg[U][4][nb] (fp64) for the nb key blocks this CTA owns, plus an fp32 copy that
// the log-sum-exp uses as a filter.  When the 4*U*n2 logits of a row group do not fit one CTA's shared
// memory, CL CTAs of a thread-block cluster split the key blocks and merge their per-row (max, sum)
// pairs through distributed shared memory.
// One sequence of the launch (a single problem is one): its representatives, scores, sizes, and key blocks per CTA.
template <typename T> struct ScoreSeq {
  const T *Qmax, *Qmin, *Kmax, *Kmin;
  const double* S_prev;
  double* S_out;
  int n1, n2, nb, cta_begin;
};
template <typename T, int NS> struct ScoreArgs { ScoreSeq<T> s[NS]; int n; };

template <typename T, int D, int U, int NS, int kThreads>
__global__ void __launch_bounds__(kThreads, kThreadsFew / kThreads)
score_kernel(const __grid_constant__ ScoreArgs<T, NS> a, int Hq, int g, int seg, int blk, double est_scale, double ln_alpha,
             double ln_1m_alpha, int fuse, int mask_first, int CL, double* stats_out) {
  constexpr int kWarps = kThreads / 32;
  extern __shared__ double smem[];
  int si = 0;
  while (NS > 1 && si + 1 < a.n && int(blockIdx.x) >= a.s[si + 1].cta_begin) ++si;
  const ScoreSeq<T>& sq = a.s[NS > 1 ? si : 0];
  const T *Qmax = sq.Qmax, *Qmin = sq.Qmin, *Kmax = sq.Kmax, *Kmin = sq.Kmin;
  const double* S_prev = sq.S_prev;
  double* S_out = sq.S_out;
  const int n1 = sq.n1, n2 = sq.n2, nb = sq.nb;
  const int cta = int(blockIdx.x) - sq.cta_begin;
  double* lg = smem;                                // [U][4][nb]
  float* lf = reinterpret_cast<float*>(smem + 4 * U * nb);   // the same logits rounded to fp32: a cheap filter for the log-sum-exp
  __shared__ double stat[4 * U];
  __shared__ double2 part[4 * U];                   // this CTA's (max, sum exp) per logit row

  // cluster rank -> owned key blocks [b_lo, b_lo + nloc)
  const int rank = CL > 1 ? cta % CL : 0;
  const int b_lo = rank * nb;
  const int nloc = max(0, min(n2, b_lo + nb) - b_lo);

  // CTA -> (b, kv head, head subgroup, segment)
  const int groups = g / U;
  int x = cta / CL;
  const int j = x % n1; x /= n1;
  const int sub = x % groups; x /= groups;
  const int kvh = x;                                 // b*Hkv + kv head
  const int Hkv = Hq / g;
  const int b = kvh / Hkv;
  const int h0 = (kvh % Hkv) * g + sub * U;          // first query head of this CTA
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto unit_of = [&](int u) { return (size_t(b) * Hq + h0 + u) * n1 + j; };

  // blocks that start at or after the end of the segment are masked (line 13)
  const int visible = min(n2, ((j + 1) * seg + blk - 1) / blk);
  // The table of ln(1 + e^-x) goes to shared memory while the predecessor ends.  Where two CTAs share an SM there is no room for it beside the B
  // operand: it is read here, and goes to the operand's place when the products are done.
  constexpr bool kShared = kThreads == kThreadsMany;
  constexpr int kTabPer = (kSpIntervals * kSpCoef + kThreads - 1) / kThreads;
  __shared__ __align__(16) double sp_tab[kSpIntervals * kSpStride];
  double tab[kTabPer];
  auto put_table = [&] {
#pragma unroll
    for (int i = 0; i < kTabPer; ++i) {
      const int e = threadIdx.x + i * kThreads;
      if (e < kSpIntervals * kSpCoef) sp_tab[(e / kSpCoef) * kSpStride + e % kSpCoef] = tab[i];
    }
  };
#pragma unroll
  for (int i = 0; i < kTabPer; ++i) tab[i] = kSoftplusTable[min(int(threadIdx.x) + i * kThreads, kSpIntervals * kSpCoef - 1)];
  if constexpr (!kShared) put_table();
  pdl_trigger();
  pdl_wait(Qmax, Qmin, Kmax, Kmin, S_prev);
  const T* kmx_base = Kmax + size_t(kvh) * n2 * D;
  const T* kmn_base = Kmin + size_t(kvh) * n2 * D;

  // The 8 x n2 x D logit products run on the fp64 tensor cores as mma.m16n8k16 with the key blocks on the
  // M side: per warp tile, A = 16 key blocks x 16 channels (streamed from the summaries, widened to fp64),
  // B = 16 channels x 8 columns, the columns being (head u, representative) = (u0 max, u0 min, u1 max, ...),
  // C = 16 blocks x 8 columns.  Lane (grp = lane/4, tig = lane%4) supplies A[grp | grp+8][c*4+tig],
  // B[i*4+tig][grp] and owns C[grp | grp+8][2*tig + {0,1}].  The channel order inside a dot product is
  // free, so lane tig takes the D/4 contiguous channels [tig*D/4, (tig+1)*D/4) of a summary row, four of
  // them per MMA: 16-byte loads, and each key value is converted once per CTA.
  constexpr int KS = D / 4;                 // channels per lane slice
  constexpr int CE = 16 / sizeof(T);        // elements per 16-byte load
  constexpr int NCH = KS / CE;              // loads per slice
  constexpr int SPC = CE / 4;               // MMA k-steps per load
  constexpr int QS = D + 2;                 // row stride of qs in doubles (odd number of 16-byte units: conflict-free)
  static_assert(8 * QS <= kSpIntervals * kSpStride, "the B operand fits where the table goes");
  __shared__ __align__(16) double qs_own[kShared ? 1 : 8 * QS];
  double* qs = kShared ? sp_tab : qs_own;   // B operand, row = column index n, laid out [k-step][tig][4 channels]
  const int tig = lane & 3, grp = lane >> 2;
  if (fuse && (lane & 15) == 0) {
    // the previous layer's scores of this CTA's elements are read once, at the very end: start them towards L2 now
    for (int u = 0; u < U; ++u)
      for (int lb = tid; lb < nloc && b_lo + lb < visible; lb += kThreads)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(S_prev + unit_of(u) * n2 + b_lo + lb));
  }
  for (int e = tid; e < 8 * D; e += kThreads) {
    const int n = e / D, ch = e % D;        // column n = (head n/2, representative n%2); channel ch
    const int u = n >> 1, rep = n & 1;
    const int tq = ch / KS, within = ch % KS;                         // owner lane-in-quad, position in its slice
    const double v = u < U ? to_f64(((rep == 0 ? Qmax : Qmin) + unit_of(u) * D)[ch]) : 0.0;
    qs[n * QS + ((within >> 2) * 4 + tq) * 4 + (within & 3)] = v;
  }
  __syncthreads();
  const int n_tiles = (nloc + 15) / 16;
  for (int t = warp; t < n_tiles; t += kWarps) {
    if (mask_first && b_lo + t * 16 >= visible) {
      // normalising over the visible blocks only: a tile of future blocks needs no products at all
      for (int e = lane; e < 4 * U * 16; e += 32) {
        const int lb = t * 16 + (e & 15);
        if (lb < nloc) { lg[(e >> 4) * nb + lb] = -CUDART_INF; lf[(e >> 4) * nb + lb] = -CUDART_INF_F; }
      }
      continue;
    }
    // this lane's two A rows (clamped in a ragged last tile), for the max and the min summaries
    const int blk0 = b_lo + min(t * 16 + grp, nloc - 1), blk1 = b_lo + min(t * 16 + grp + 8, nloc - 1);
    const uint4* src[4] = {reinterpret_cast<const uint4*>(kmx_base + size_t(blk0) * D + tig * KS),
                           reinterpret_cast<const uint4*>(kmx_base + size_t(blk1) * D + tig * KS),
                           reinterpret_cast<const uint4*>(kmn_base + size_t(blk0) * D + tig * KS),
                           reinterpret_cast<const uint4*>(kmn_base + size_t(blk1) * D + tig * KS)};
    double cx[4] = {0.0, 0.0, 0.0, 0.0}, cn[4] = {0.0, 0.0, 0.0, 0.0};
    uint4 cur[4], nxt[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) cur[i] = __ldg(src[i]);
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
      if (ch + 1 < NCH) {
#pragma unroll
        for (int i = 0; i < 4; ++i) nxt[i] = __ldg(src[i] + ch + 1);
      }
#pragma unroll
      for (int sp = 0; sp < SPC; ++sp) {
        const int step = ch * SPC + sp;
        double ax[8], an[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          ax[2 * c] = to_f64(reinterpret_cast<const T*>(&cur[0])[sp * 4 + c]);
          ax[2 * c + 1] = to_f64(reinterpret_cast<const T*>(&cur[1])[sp * 4 + c]);
          an[2 * c] = to_f64(reinterpret_cast<const T*>(&cur[2])[sp * 4 + c]);
          an[2 * c + 1] = to_f64(reinterpret_cast<const T*>(&cur[3])[sp * 4 + c]);
        }
        const double2 b01 = *reinterpret_cast<const double2*>(&qs[grp * QS + (step * 4 + tig) * 4]);
        const double2 b23 = *reinterpret_cast<const double2*>(&qs[grp * QS + (step * 4 + tig) * 4 + 2]);
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7,%8,%9,%10,%11}, "
            "{%12,%13,%14,%15}, {%0,%1,%2,%3};"
            : "+d"(cx[0]), "+d"(cx[1]), "+d"(cx[2]), "+d"(cx[3])
            : "d"(ax[0]), "d"(ax[1]), "d"(ax[2]), "d"(ax[3]), "d"(ax[4]), "d"(ax[5]), "d"(ax[6]), "d"(ax[7]),
              "d"(b01.x), "d"(b01.y), "d"(b23.x), "d"(b23.y));
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7,%8,%9,%10,%11}, "
            "{%12,%13,%14,%15}, {%0,%1,%2,%3};"
            : "+d"(cn[0]), "+d"(cn[1]), "+d"(cn[2]), "+d"(cn[3])
            : "d"(an[0]), "d"(an[1]), "d"(an[2]), "d"(an[3]), "d"(an[4]), "d"(an[5]), "d"(an[6]), "d"(an[7]),
              "d"(b01.x), "d"(b01.y), "d"(b23.x), "d"(b23.y));
      }
      if (ch + 1 < NCH) {
#pragma unroll
        for (int i = 0; i < 4; ++i) cur[i] = nxt[i];
      }
    }
    // C[i]: block grp + 8*(i/2), column 2*tig + (i%2) = (head tig, representative i%2);
    // representative 0 (Qmax): cx = l1, cn = l2; representative 1 (Qmin): cx = l3, cn = l4
    if (tig < U) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int lb = t * 16 + grp + (i >> 1) * 8;      // local block index
        const int rep = i & 1;
        if (lb < nloc) {
          const bool hide = mask_first && b_lo + lb >= visible;
          const double vx = hide ? -CUDART_INF : cx[i] * est_scale, vn = hide ? -CUDART_INF : cn[i] * est_scale;
          lg[(tig * 4 + rep * 2 + 0) * nb + lb] = vx;
          lg[(tig * 4 + rep * 2 + 1) * nb + lb] = vn;
          lf[(tig * 4 + rep * 2 + 0) * nb + lb] = float(vx);
          lf[(tig * 4 + rep * 2 + 1) * nb + lb] = float(vn);
        }
      }
    }
  }
  __syncthreads();
  if constexpr (kShared) put_table();

  // log-sum-exp of each of the 4U logit rows (softmax over blocks, lines 9-10): a warp owns a row, so only
  // shuffles are needed.  Terms more than e^-50 below the row maximum cannot change the rounded sum and
  // are skipped.  Only a few percent of a row survive that test, scattered over the lanes, so the row is
  // first scanned in fp32 and the candidates -- fp32 value within 50 + a rounding margin of the fp32
  // maximum, which always includes the true maximum and every term that counts -- are compacted into a
  // dense index list (in place, over the fp32 row); the fp64 maximum and the exponentials then run on full warps.
#pragma unroll 1
  for (int rI = warp; rI < 4 * U; rI += kWarps) {
    const double* rowp = lg + rI * nb;
    float* rowf = lf + rI * nb;
    float mf = -CUDART_INF_F;
#pragma unroll 4
    for (int lb = lane; lb < nloc; lb += 32) mf = fmaxf(mf, rowf[lb]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
    const float thr = mf - (51.0f + fabsf(mf) * 1e-6f);     // -inf when the whole (local) row is masked: no candidates
    int* cand = reinterpret_cast<int*>(rowf);                // entry i is written after element i has been read
    int ncand = 0;
    for (int base = 0; base < nloc; base += 32) {
      const int lb = base + lane;
      const bool c = lb < nloc && rowf[lb] > thr;
      const unsigned ballot = __ballot_sync(0xffffffffu, c);
      if (c) cand[ncand + __popc(ballot & ((1u << lane) - 1u))] = lb;
      ncand += __popc(ballot);
    }
    __syncwarp();
    double m = -CUDART_INF;
    for (int i = lane; i < ncand; i += 32) m = fmax(m, rowp[cand[i]]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    double sum = 0.0;
    for (int i = lane; i < ncand; i += 32) {
      const double d = rowp[cand[i]] - m;
      if (d > -50.0) sum += exp(d);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) part[rI] = make_double2(m, sum);
  }
  __syncthreads();
  if (CL > 1) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();                                   // every CTA's partials are in place
    // thread (row, r) fetches rank r's pair of that row; the CL lanes of a row are adjacent, so the merge is shuffles
    if (warp * 32 < 4 * U * CL) {                     // whole warps take part in the shuffles
      const bool act = tid < 4 * U * CL;
      const int row = act ? tid / CL : 0, r = tid % CL;
      const double2 pr = cluster.map_shared_rank(part, r)[row];
      double M = pr.x;
      for (int o = CL >> 1; o > 0; o >>= 1) M = fmax(M, __shfl_xor_sync(0xffffffffu, M, o));
      double Ssum = pr.y > 0.0 ? pr.y * exp(pr.x - M) : 0.0;
      for (int o = CL >> 1; o > 0; o >>= 1) Ssum += __shfl_xor_sync(0xffffffffu, Ssum, o);
      if (act && r == 0) stat[row] = M + log(Ssum);
    }
    // no CTA may exit while a peer can still read its partials: arrive now, wait at the end of the kernel
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  } else if (tid < 4 * U) {
    stat[tid] = part[tid].x + log(part[tid].y);
  }
  __syncthreads();

  // stats_out given: this launch only produces the four log-sum-exps of every (head, segment) row
  if (stats_out != nullptr && rank == 0 && tid < 4 * U) stats_out[unit_of(tid >> 2) * 4 + (tid & 3)] = stat[tid];

  // combine (lines 11-12), mask (13), fusion (14) over this CTA's blocks of the U rows
  const double ln2 = 0.693147180559945309417232121458;
#pragma unroll 1
  for (int u = 0; u < (stats_out != nullptr ? 0 : U); ++u) {
    const double* l = lg + u * 4 * nb;
    const double st1 = stat[u * 4 + 0], st2 = stat[u * 4 + 1], st3 = stat[u * 4 + 2], st4 = stat[u * 4 + 3];
    const size_t out_row = unit_of(u) * n2 + b_lo;
#pragma unroll 2
    for (int lb = tid; lb < nloc; lb += kThreads) {
      double v;
      if (b_lo + lb >= visible) {
        v = -CUDART_INF;
      } else {
        const double L1 = l[lb] - st1, L2 = l[nb + lb] - st2, L3 = l[2 * nb + lb] - st3, L4 = l[3 * nb + lb] - st4;
        // max( ln (S1+S3)/2, ln (S2+S4)/2 ).  ln(e^a + e^b) lies in [max(a,b), max(a,b) + ln 2], so the pair with the
        // larger maximum wins outright unless the two maxima are within ln 2 of each other: one evaluation, rarely two.
        const double h13 = fmax(L1, L3), h24 = fmax(L2, L4);
        const bool first = h13 >= h24;
        v = logaddexp(first ? L1 : L2, first ? L3 : L4, sp_tab);
        if (fabs(h13 - h24) < ln2) v = fmax(v, logaddexp(first ? L2 : L1, first ? L4 : L3, sp_tab));
        v -= ln2;
        if (fuse) v = logaddexp(ln_alpha + v, ln_1m_alpha + S_prev[out_row + lb], sp_tab);
      }
      S_out[out_row + lb] = v;
    }
  }
  if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Key blocks are split over a cluster of 1, 2, 4 or 8 CTAs until one fits an SM (200 KB of logits each), and twice as often where two then fit
// an SM (104 KB) and that is the faster split; 0: 8 are not enough.  With 4 heads it is the faster one only while all CTAs run at once:
// 552 < n2 <= 1064, one CTA with 512 threads / two of half the blocks, us, in graphs, bf16: 5 segments x 8 KV heads, n2 600 25.6 / 16.4; 15 x 8,
// n2 938 33.2 / 37.0; 34 x 8, n2 576 46.0 / 52.1; 145 x 8, n2 580 10 to 12 % slower split.  With 1 or 2 heads, whose MMAs are a quarter or half empty
// columns, the split is never slower: 30 x 8, 2 heads, n2 1132 65.9 / 65.8 (64 channels 52.1 / 48.1); 25 x 12, one head, n2 2268 119.4 / 95.2.
constexpr size_t kSmemShared = 104 * 1024, kSmemWideRows = 88 * 1024 + 512, kSmemAlone = 200 * 1024;
int cluster_of(const Dims& m, int U, int* nb) {
  auto split = [&](int CL) {
    *nb = (((m.n2 + CL - 1) / CL) + 7) & ~7;
    return (sizeof(double) + sizeof(float)) * 4 * size_t(U) * *nb;
  };
  int CL = 1;
  while (split(CL) > kSmemAlone)
    if ((CL *= 2) > 8) return 0;
  const bool twice = CL < 8 && split(CL) > kSmemShared && split(2 * CL) <= kSmemShared &&
                     (U < 4 || (long long)m.B * m.Hkv * (m.g / U) * m.n1 * 2 * CL <= 148);
  if (twice) CL *= 2;
  split(CL);
  return CL;
}
// CTAs of 256 threads, two per SM, where there are more of them than SMs (see kThreadsMany).  Rows of 512 bytes (fp32, 128 channels) need
// the L1 that two CTAs of more than 88.5 KB (196 KB of the SM with their static part) leave no room for: n2 464 / 480, 34 / 32 segments x 8 KV
// heads, one CTA 55.1 / 55.4 us, two 54.2 / 71.2.
bool two_per_sm(const Dims& m, long long ctas, size_t smem) { return ctas > 148 && smem <= (m.d * m.es == 512 ? kSmemWideRows : kSmemShared); }
struct ScoreProblem { Dims m; const char* ws; const double* S_prev; double* S_out; };

// problems that need the same cluster size, in one launch
template <typename T, int D, int U, int NS>
int launch_u(const cp_params& p, const ScoreProblem* pr, int n, int CL, double* stats_out, cudaStream_t st) {
  ScoreArgs<T, NS> a;
  a.n = n;
  long long ctas = 0;
  int nb_max = 0;
  for (int i = 0; i < n; ++i) {
    const Dims& m = pr[i].m;
    const WsLayout w = ws_layout(m);
    ScoreSeq<T>& s = a.s[i];
    s.Qmax = reinterpret_cast<const T*>(pr[i].ws + w.qmax); s.Qmin = reinterpret_cast<const T*>(pr[i].ws + w.qmin);
    s.Kmax = reinterpret_cast<const T*>(pr[i].ws + w.kmax); s.Kmin = reinterpret_cast<const T*>(pr[i].ws + w.kmin);
    s.S_prev = pr[i].S_prev; s.S_out = pr[i].S_out; s.n1 = m.n1; s.n2 = m.n2;
    cluster_of(m, U, &s.nb);
    if (s.nb > nb_max) nb_max = s.nb;
    if (ctas > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
    s.cta_begin = int(ctas);
    ctas += (long long)m.B * m.Hkv * (m.g / U) * m.n1 * CL;
  }
  if (ctas > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  const Dims& m = pr[0].m;
  const size_t smem = (sizeof(double) + sizeof(float)) * (4 * size_t(U) * nb_max);   // fp64 logits + their fp32 copies
  const bool many = two_per_sm(m, ctas, smem);
  auto kern = many ? score_kernel<T, D, U, NS, kThreadsMany> : score_kernel<T, D, U, NS, kThreadsFew>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
    return CP_ERR_CUDA;
  const double al = double(p.alpha);
  const int fuse = (pr[0].S_prev != nullptr && p.alpha != 1.0f) ? 1 : 0, mask_first = (p.flags & CP_FLAG_MASK_BEFORE_SOFTMAX) ? 1 : 0;
  return launch_pdl_cluster(kern, dim3(unsigned(ctas)), many ? kThreadsMany : kThreadsFew, smem, unsigned(CL), st, a, m.Hq, m.g, m.seg, m.blk,
                            double(p.est_scale), log(al), log1p(-al), fuse, mask_first, CL, stats_out);
}

template <typename T, int D, int NS>
int launch_t(const cp_params& p, const ScoreProblem* pr, int n, int CL, double* stats_out, cudaStream_t st) {
  const int U = score_heads(pr[0].m);
  if (U == 4) return launch_u<T, D, 4, NS>(p, pr, n, CL, stats_out, st);
  if (U == 2) return launch_u<T, D, 2, NS>(p, pr, n, CL, stats_out, st);
  return launch_u<T, D, 1, NS>(p, pr, n, CL, stats_out, st);
}

template <int NS>
int launch_problems(const cp_params& p, const ScoreProblem* pr, int n, int CL, double* stats_out, cudaStream_t st) {
  const int d = pr[0].m.d;
  if (p.dtype == CP_BF16) {
    if (d == 128) return launch_t<__nv_bfloat16, 128, NS>(p, pr, n, CL, stats_out, st);
    if (d == 64) return launch_t<__nv_bfloat16, 64, NS>(p, pr, n, CL, stats_out, st);
  } else if (p.dtype == CP_F16) {
    if (d == 128) return launch_t<__half, 128, NS>(p, pr, n, CL, stats_out, st);
    if (d == 64) return launch_t<__half, 64, NS>(p, pr, n, CL, stats_out, st);
  } else {
    if (d == 128) return launch_t<float, 128, NS>(p, pr, n, CL, stats_out, st);
    if (d == 64) return launch_t<float, 64, NS>(p, pr, n, CL, stats_out, st);
  }
  return CP_ERR_UNSUPPORTED;
}

}  // namespace

// The general kernel: any dtype, head_dim 64 or 128.  With stats_out it only writes the four log-sum-exps
// of every (head, segment) row, [B,Hq,n1,4], and leaves S_out alone.
int launch_score_generic(const cp_params& p, const Dims& m, const char* ws, const double* S_prev,
                         double* S_out, double* stats_out, cudaStream_t st) {
  const ScoreProblem pr{m, ws, S_prev, S_out};
  int nb;
  const int CL = cluster_of(m, score_heads(m), &nb);
  return CL == 0 ? CP_ERR_UNSUPPORTED : launch_problems<1>(p, &pr, 1, CL, stats_out, st);
}

int launch_score_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, char* const* ws, int n_seqs, const double* S_prev,
                      double* S_out, cudaStream_t st) {
  int nb;
  for (int CL = 1; CL <= 8; CL *= 2) {
    ScoreProblem pr[kSeqsPerLaunch];
    int n = 0;
    for (int i = 0; i <= n_seqs; ++i) {
      if (n == kSeqsPerLaunch || (i == n_seqs && n > 0)) {
        const int rc = launch_problems<kSeqsPerLaunch>(p, pr, n, CL, nullptr, st);
        if (rc != CP_OK) return rc;
        n = 0;
      }
      if (i == n_seqs) break;
      const Dims q = seq_dims(m, slots[i].len);
      const int c = cluster_of(q, score_heads(q), &nb);
      if (c == 0) return CP_ERR_UNSUPPORTED;
      if (c == CL) pr[n++] = {q, ws[i], S_prev ? S_prev + slots[i].s : nullptr, S_out + slots[i].s};
    }
  }
  return CP_OK;
}

}  // namespace cp
