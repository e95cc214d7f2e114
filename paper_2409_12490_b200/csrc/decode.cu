// Block criticality of the newest token (Algorithm 1 on a segment that holds one token: Qmax = Qmin = q), 16- or 32-bit keys.
//
// The key cache is read once: a warp takes a key block, folds its rows into the per-channel max and min in registers and multiplies them with
// the group's queries in fp64 right there, so the representatives never go to memory and every SM takes part.  A head's two rows of
// logits are then normalised: ln S = max(l1 - lse1, l2 - lse2).  Short rows: all of it in decode_rows_kernel, one launch.  Others: the
// logits go to memory (decode_logits_kernel) and decode_score_kernel takes a head each.  The general kernels, which take what is left, write
// the representatives and score each KV head's whole cache on one cluster of CTAs (130001 tokens, 8 KV heads, block 128: the two calls
// 110 us, here 53; 41 us is the read of K at the copy rate, which bounds it).
#include <math_constants.h>

#include <algorithm>

#include "score_common.cuh"
#include "summarize.cuh"

namespace cp {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxCluster = 16, kMaxRowWarps = 16;

// decode_rows_kernel's shape: a cluster of `ctas` CTAs of `warps` warps per KV head, `slots` blocks per CTA.
struct RowShape { int warps, slots, ctas; };

// Rows of up to 256 blocks (16 CTAs of 16 warps) and groups of up to 8 heads take decode_rows_kernel: a launch less (3.4 us of host work against
// 5.7) and no trip of the logits through memory.  Both calls of a token, us, in a graph over cold keys, blocks of 32 rows, 4 heads per KV head,
// two kernels / one: 8 KV heads: 256 blocks 16.5 / 13.2, 125 12.4 / 10.9, 32 9.9 / 8.8; 56: 63 blocks 18.4 / 16.8, 32 16.2 / 13.9; where the host
// launches them 22 / 20.  More heads make products in fp64 the larger part, which too few SMs share (1 KV head: 16 heads, 63 blocks 12.5 / 14.9;
// 8 heads, 32 blocks 7.4 / 7.5).  With many thousand blocks (B x KV heads x n2) the chip is full anyway, and single CTAs that come and go keep it
// fuller than clusters (14336 37.8 / 35.2, 65536 114 / 118).
// A block per warp while all CTAs are resident at once (64 registers a thread; clusters of more than 8 CTAs leave about a third of the
// chip's places empty, as each has to lie within one part of it); beyond, two blocks one after the other, if they are long enough to hide that.
// One / two, us: 256 blocks: 8 KV heads 13.1 / 15.2, 12 14.8 / 16.2, 16 20.9 / 17.5, 24 23.8 / 19.6; 125 blocks: 16 13.7 / 13.9, 24 15.4 / 15.0, 32 19.6 /
// 17.3; 32 blocks: 128 17.2 / 18.4, 256 28.6 / 25.1.  Two kernels / two: 256 blocks, 56 KV heads: 32 rows of 256 bytes 37.8 / 35.2, 16 24.2 / 26.5.
bool rows_in_one_launch(const Dims& m, RowShape* s) {
  if (m.n2 > kMaxCluster * kMaxRowWarps || m.g > 8 || (long long)m.B * m.Hkv * m.n2 > 16384) return false;
  s->warps = std::max(kWarps, (m.n2 + kMaxCluster - 1) / kMaxCluster);
  s->slots = s->warps;
  s->ctas = (m.n2 + s->slots - 1) / s->slots;
  const int places = (32 / s->warps) * (s->ctas > 8 ? 148 * 2 / 3 : 148);
  if ((long long)m.B * m.Hkv * s->ctas <= places) return true;
  s->slots *= 2;
  s->ctas = (m.n2 + s->slots - 1) / s->slots;
  return m.blk * m.d * m.es >= 8192;
}

// Per-channel max and min of the rows of a block, in the LPR lanes of every group of lanes
template <typename T, int LPR>
__device__ __forceinline__ void scan_block(const char* base, int64_t st_bytes, int rows, int lane, uint4& mx, uint4& mn) {
  scan_rows<T, LPR>(base, st_bytes, 0, rows, 32 / LPR, lane, mx, mn);
#pragma unroll
  for (int m = LPR; m < 32; m <<= 1) { uint4 o = shfl_xor4(mx, m); vmax<T>(mx, o); o = shfl_xor4(mn, m); vmin<T>(mn, o); }
}
// (head u, max | min) products, dealt to the lane groups that hold a copy of the representatives each: out(2 u + is_min, logit)
template <typename T, int LPR, typename Out>
__device__ __forceinline__ void block_logits(const T* qs, int g, const uint4& mx, const uint4& mn, int lane, double est_scale, Out out) {
  constexpr int CE = 16 / int(sizeof(T));          // channels per lane
  constexpr int SUBS = 32 / LPR;
  const int sub = lane / LPR, col = lane % LPR;
#pragma unroll 1
  for (int t0 = 0; t0 < 2 * g; t0 += SUBS) {
    const int t = t0 + sub;
    const uint4 kv = (t & 1) ? mn : mx, qv = reinterpret_cast<const uint4*>(qs)[min(t >> 1, g - 1) * LPR + col];
    const T *ke = reinterpret_cast<const T*>(&kv), *qe = reinterpret_cast<const T*>(&qv);
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int i = 0; i < CE; i += 2) {
      s0 = fma(to_f64(qe[i]), to_f64(ke[i]), s0);
      s1 = fma(to_f64(qe[i + 1]), to_f64(ke[i + 1]), s1);
    }
    s0 += s1;
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    if (col == 0 && t < 2 * g) out(t, s0 * est_scale);
  }
}

template <typename T, int LPR>
__global__ void __launch_bounds__(kThreads, 5)
decode_logits_kernel(const T* __restrict__ q_last, const char* __restrict__ K, int64_t sb, int64_t sh, int64_t st, int Hkv, int g, int n,
                     int blk, int n2, double est_scale, double* l_max, double* l_min) {
  constexpr int D = LPR * 16 / int(sizeof(T));
  extern __shared__ __align__(16) uint8_t smem[];
  T* qs = reinterpret_cast<T*>(smem);              // [g][D]
  pdl_trigger();
  pdl_wait(q_last, K);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kvh = blockIdx.y, b = kvh / Hkv;       // b * Hkv + kv head
  const int h0 = kvh * g;                          // b * Hq + first query head of the group
  for (int e = threadIdx.x; e < g * LPR; e += kThreads)
    reinterpret_cast<uint4*>(qs)[e] = __ldg(reinterpret_cast<const uint4*>(q_last + size_t(h0) * D) + e);
  const int bb = blockIdx.x * kWarps + warp;
  uint4 mx, mn;
  if (bb < n2) {
    const char* base = K + (int64_t(b) * sb + int64_t(kvh % Hkv) * sh + int64_t(bb) * blk * st) * int(sizeof(T));
    scan_block<T, LPR>(base, st * int(sizeof(T)), min(blk, n - bb * blk), lane, mx, mn);
  }
  __syncthreads();
  if (bb >= n2) return;
  block_logits<T, LPR>(qs, g, mx, mn, lane, est_scale,
                       [&](int t, double l) { ((t & 1) ? l_min : l_max)[size_t(h0 + (t >> 1)) * n2 + bb] = l; });
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// scale * exp(l - m) as the normalisations take it: terms below e^-50 of the largest cannot change the rounded sum; NaN stays out
__device__ __forceinline__ double term(double l, double m, double scale) { return l - m > -50.0 ? scale * exp(l - m) : 0.0; }

// Short rows in one launch: a cluster of up to 16 CTAs per KV head, one block or two per warp.  The logits stay in shared memory; a CTA gives the
// (max, sum) of its blocks to the others through distributed shared memory, all merge them in the same order, and each writes its blocks' ln S.
template <typename T, int LPR>
__global__ void __launch_bounds__(kMaxRowWarps * 32, 2)
decode_rows_kernel(const T* __restrict__ q_last, const char* __restrict__ K, int64_t sb, int64_t sh, int64_t st, int Hkv, int g, int n,
                   int blk, int n2, int slots, double est_scale, double* __restrict__ S) {
  constexpr int D = LPR * 16 / int(sizeof(T));
  extern __shared__ __align__(16) uint8_t smem[];
  const int warps = blockDim.x >> 5, ctas = gridDim.x, rank = blockIdx.x;       // a cluster is a row of the grid
  double2* part = reinterpret_cast<double2*>(smem);                             // [CTA][2 g]: (max, sum) of its blocks
  double* rows = reinterpret_cast<double*>(part + ctas * 2 * g);                // [2 g][slots]
  double* lse = rows + 2 * g * slots;                                           // [2 g]
  T* qs = reinterpret_cast<T*>(lse + 2 * g);                                    // [g][D]
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");         // this CTA has started: the others may write to part
  pdl_trigger();
  pdl_wait(q_last, K);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kvh = blockIdx.y, b = kvh / Hkv, h0 = kvh * g;
  for (int e = threadIdx.x; e < g * LPR; e += blockDim.x)
    reinterpret_cast<uint4*>(qs)[e] = __ldg(reinterpret_cast<const uint4*>(q_last + size_t(h0) * D) + e);
  __syncthreads();
  const int b0 = rank * slots, nb = min(slots, n2 - b0);                        // this CTA's blocks
  const char* base = K + (int64_t(b) * sb + int64_t(kvh % Hkv) * sh) * int(sizeof(T));
#pragma unroll 1
  for (int w = warp; w < nb; w += warps) {
    uint4 mx, mn;
    const int t0 = (b0 + w) * blk;
    scan_block<T, LPR>(base + int64_t(t0) * st * int(sizeof(T)), st * int(sizeof(T)), min(blk, n - t0), lane, mx, mn);
    block_logits<T, LPR>(qs, g, mx, mn, lane, est_scale, [&](int t, double l) { rows[t * slots + w] = l; });
  }
  __syncthreads();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  for (int r = warp; r < 2 * g; r += warps) {
    const double l = lane < nb ? rows[r * slots + lane] : -CUDART_INF;
    const double m = warp_max(l);
    const double s = warp_sum(term(l, m, 1.0));
    if (lane < ctas) {
      uint32_t to;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(uint32_t(__cvta_generic_to_shared(part + rank * 2 * g + r))), "r"(lane));
      asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(to), "d"(m), "d"(s) : "memory");
    }
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  for (int r = warp; r < 2 * g; r += warps) {
    const double2 p = lane < ctas ? part[lane * 2 * g + r] : make_double2(-CUDART_INF, 0.0);
    const double m = warp_max(p.x);
    const double s = warp_sum(term(p.x, m, p.y));
    // Logits that are not finite end as in score_kernel: a row without a finite maximum has the sum 0 and ln 0 = -inf
    if (lane == 0) lse[r] = s > 0.0 ? m + log(s) : -CUDART_INF;
  }
  __syncthreads();
  for (int x = threadIdx.x; x < g * nb; x += blockDim.x) {
    const int u = x / nb, w = x % nb;
    const double L1 = rows[2 * u * slots + w] - lse[2 * u], L2 = rows[(2 * u + 1) * slots + w] - lse[2 * u + 1];
    S[size_t(h0 + u) * n2 + b0 + w] = L1 >= L2 ? L1 : L2;
  }
}

// One CTA per (batch, head): S[row] holds the Kmax logits on entry and ln S on return; l_min the Kmin logits.
template <int NPT>
__global__ void __launch_bounds__(kThreads)
decode_score_kernel(double* __restrict__ S, const double* __restrict__ l_min, int n2) {
  __shared__ double2 red[kWarps];
  pdl_trigger();
  pdl_wait(S, l_min);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* row = S + size_t(blockIdx.x) * n2;
  const double* row2 = l_min + size_t(blockIdx.x) * n2;
  double a[NPT], c[NPT];
  double2 m = make_double2(-CUDART_INF, -CUDART_INF);
#pragma unroll
  for (int i = 0; i < NPT; ++i) {
    const int x = tid + i * kThreads;
    a[i] = x < n2 ? row[x] : -CUDART_INF;
    c[i] = x < n2 ? row2[x] : -CUDART_INF;
    m.x = fmax(m.x, a[i]); m.y = fmax(m.y, c[i]);
  }
  auto block_reduce = [&](double2 v, bool is_max) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, v.x, o), y = __shfl_xor_sync(0xffffffffu, v.y, o);
      v.x = is_max ? fmax(v.x, x) : v.x + x; v.y = is_max ? fmax(v.y, y) : v.y + y;
    }
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = red[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      v.x = is_max ? fmax(v.x, red[w].x) : v.x + red[w].x; v.y = is_max ? fmax(v.y, red[w].y) : v.y + red[w].y;
    }
    __syncthreads();
    return v;
  };
  m = block_reduce(m, true);
  double2 s = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int i = 0; i < NPT; ++i) {                  // terms below e^-50 of the largest cannot change the rounded sum; NaN stays out
    if (tid + i * kThreads >= n2) break;
    double av = a[0], cv = c[0];
#pragma unroll
    for (int x = 1; x < NPT; ++x) { av = x == i ? a[x] : av; cv = x == i ? c[x] : cv; }
    if (av - m.x > -50.0) s.x += exp(av - m.x);
    if (cv - m.y > -50.0) s.y += exp(cv - m.y);
  }
  s = block_reduce(s, false);
  // Logits that are not finite end as in score_kernel, which larger blocks go through: a NaN logit is the NaN of its own block
  // alone, and a row without a finite maximum has the sum 0 and ln 0 = -inf.
  const double lse1 = s.x > 0.0 ? m.x + log(s.x) : -CUDART_INF, lse2 = s.y > 0.0 ? m.y + log(s.y) : -CUDART_INF;
#pragma unroll
  for (int i = 0; i < NPT; ++i) {
    const int x = tid + i * kThreads;
    const double L1 = a[i] - lse1, L2 = c[i] - lse2;
    if (x < n2) row[x] = L1 >= L2 ? L1 : L2;
  }
}

template <typename T, int LPR>
int launch_logits(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* l_max, double* l_min, cudaStream_t st) {
  const dim3 grid(unsigned((m.n2 + kWarps - 1) / kWarps), unsigned(m.B * m.Hkv));
  const size_t smem = size_t(m.g) * m.d * m.es;    // the group's queries: up to 64 KB (fp32, 128 channels, 128 heads)
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(decode_logits_kernel<T, LPR>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
    return CP_ERR_CUDA;
  return launch_pdl(decode_logits_kernel<T, LPR>, grid, kThreads, smem, st, static_cast<const T*>(q_last),
                    static_cast<const char*>(K), p.k_stride[0], p.k_stride[1], p.k_stride[2], m.Hkv, m.g, m.n, m.blk, m.n2,
                    double(p.est_scale), l_max, l_min);
}

template <typename T, int LPR>
int launch_rows(const cp_params& p, const Dims& m, const RowShape& s, const void* q_last, const void* K, double* S, cudaStream_t st) {
  const size_t rows = 2 * size_t(m.g);
  const size_t smem = s.ctas * rows * sizeof(double2) + rows * (s.slots + 1) * sizeof(double) + size_t(m.g) * m.d * m.es;   // up to 10 KB
  auto kern = decode_rows_kernel<T, LPR>;
  if (s.ctas > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return CP_ERR_CUDA;
  return launch_pdl_cluster(kern, dim3(unsigned(s.ctas), unsigned(m.B * m.Hkv)), unsigned(s.warps * 32), smem, unsigned(s.ctas), st,
                            static_cast<const T*>(q_last), static_cast<const char*>(K), p.k_stride[0], p.k_stride[1], p.k_stride[2], m.Hkv, m.g,
                            m.n, m.blk, m.n2, s.slots, double(p.est_scale), S);
}

template <typename T, int LPR>
int launch_typed(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* S_out, double* l_min, cudaStream_t st) {
  RowShape shape;
  if (rows_in_one_launch(m, &shape)) return launch_rows<T, LPR>(p, m, shape, q_last, K, S_out, st);
  const int rc = launch_logits<T, LPR>(p, m, q_last, K, S_out, l_min, st);
  if (rc != CP_OK) return rc;
  const dim3 grid(unsigned(m.B * m.Hq));
  if (m.n2 <= 4 * kThreads) return launch_pdl(decode_score_kernel<4>, grid, kThreads, 0, st, S_out, l_min, m.n2);
  if (m.n2 <= 16 * kThreads) return launch_pdl(decode_score_kernel<16>, grid, kThreads, 0, st, S_out, l_min, m.n2);
  return launch_pdl(decode_score_kernel<32>, grid, kThreads, 0, st, S_out, l_min, m.n2);
}

}  // namespace

// Blocks of up to 128 rows (a warp each), and query groups whose Kmin logits fit the workspace's key representatives
// ([B,Hkv,n2,d] twice), whose place they take: 8 g <= 2 d es, at least 32 heads per KV head.
bool decode_path_applies(const Dims& m) { return m.blk <= 128 && 8 * m.g <= 2 * m.d * m.es && m.B * (long long)m.Hkv <= 65535; }

int launch_decode_score(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* S_out, char* ws, cudaStream_t st) {
  double* l_min = reinterpret_cast<double*>(ws + ws_layout(m).kmax);
  const int lpr = m.d * m.es / 16;
  if (p.dtype == CP_BF16)
    return lpr == 16 ? launch_typed<__nv_bfloat16, 16>(p, m, q_last, K, S_out, l_min, st) : launch_typed<__nv_bfloat16, 8>(p, m, q_last, K, S_out, l_min, st);
  if (p.dtype == CP_F16)
    return lpr == 16 ? launch_typed<__half, 16>(p, m, q_last, K, S_out, l_min, st) : launch_typed<__half, 8>(p, m, q_last, K, S_out, l_min, st);
  return lpr == 32 ? launch_typed<float, 32>(p, m, q_last, K, S_out, l_min, st) : launch_typed<float, 16>(p, m, q_last, K, S_out, l_min, st);
}

}  // namespace cp
