// Block criticality of the newest token (Algorithm 1 on a segment that holds one token: Qmax = Qmin = q), 16- or 32-bit keys.
//
// decode_logits_kernel reads the key cache once: a warp takes a key block, folds its rows into the per-channel max and min in
// registers and multiplies them with the group's queries in fp64 right there, so the representatives never go to memory and
// every SM takes part.  decode_score_kernel then normalises a head's two logit rows: ln S = max(l1 - lse1, l2 - lse2).  The general
// kernels, which this replaces, wrote the representatives and scored each KV head's whole cache on one cluster of CTAs (130001
// tokens, 8 KV heads, block 128: the pass 110 us, here 55; 41 us is the read of K at the copy rate, which bounds it).
#include <math_constants.h>

#include "score_common.cuh"
#include "summarize.cuh"

namespace cp {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxFusedGroup = 32, kMaxFusedLogits = 2048;
constexpr int kMaxFusedHeads = (kStatusBytes - int(sizeof(DeviceStatus))) / int(sizeof(unsigned));   // counters behind the status word

// Rows that the logits kernel normalises itself, one launch less: those of a KV head are one CTA's work then, so it has to be little: a
// row per warp, eight values per lane.  Both calls of a token, us, 32 / 8 heads, 256 blocks, normalised by a kernel of its own / by the last
// CTA: 24.1 / 19.4 where the host launches them (that bounds both; about half of it is the launch), 12.5 / 14.7 in a graph.  1016 blocks 55.6 /
// 71.1, a head per KV head and some 1000 blocks 26.2 / 30.8 (rows read from L2 by the warps, one after another).
bool fused_rows(const Dims& m) { return m.g <= kMaxFusedGroup && m.B * m.Hkv <= kMaxFusedHeads && m.n2 <= kThreads && 2 * m.g * m.n2 <= kMaxFusedLogits; }

template <typename T, int LPR>
__global__ void __launch_bounds__(kThreads, 5)
decode_logits_kernel(const T* __restrict__ q_last, const char* __restrict__ K, int64_t sb, int64_t sh, int64_t st, int Hkv, int g, int n,
                     int blk, int n2, double est_scale, double* l_max, double* l_min, unsigned* done) {
  constexpr int CE = 16 / int(sizeof(T));          // channels per lane
  constexpr int D = LPR * CE;
  constexpr int SUBS = 32 / LPR;
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
    scan_rows<T, LPR>(base, st * int(sizeof(T)), 0, min(blk, n - bb * blk), SUBS, lane, mx, mn);
#pragma unroll
    for (int m = LPR; m < 32; m <<= 1) { uint4 o = shfl_xor4(mx, m); vmax<T>(mx, o); o = shfl_xor4(mn, m); vmin<T>(mn, o); }
  }
  __syncthreads();
  // (head u, max | min) products, dealt to the SUBS lane groups that hold a copy of the representatives each
  const int sub = lane / LPR, col = lane % LPR;
#pragma unroll 1
  for (int t0 = 0; t0 < (bb < n2 ? 2 * g : 0); t0 += SUBS) {
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
    if (col == 0 && t < 2 * g) ((t & 1) ? l_min : l_max)[size_t(h0 + (t >> 1)) * n2 + bb] = s0 * est_scale;
  }
  if (done == nullptr) return;

  // The last CTA of a KV head normalises the rows of its group (small ones: fused_rows): all of them come from L2, where the other CTAs
  // left them, in one go, a warp takes a row at a time from shared memory, and all are written in one go.
  __shared__ bool last;
  __shared__ double lse[2 * kMaxFusedGroup];
  __shared__ double rows[kMaxFusedLogits];         // [Kmax | Kmin][head][block]
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();                               // the CTA's logits, which the barrier has ordered before this, are visible
    last = atomicAdd(done + kvh, 1u) == gridDim.x - 1;
    if (last) done[kvh] = 0;                       // for the next call
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  const int gn = g * n2;
  double *out = l_max + size_t(h0) * n2, *other = l_min + size_t(h0) * n2;
#pragma unroll
  for (int i = 0; i < kMaxFusedLogits / 2 / kThreads; ++i) {
    const int x = i * kThreads + threadIdx.x;
    if (x < gn) { rows[x] = __ldcg(out + x); rows[gn + x] = __ldcg(other + x); }
  }
  __syncthreads();
  for (int r = warp; r < 2 * g; r += kWarps) {
    const double* l = rows + r * n2;
    double m = -CUDART_INF, s = 0.0;
    for (int x = lane; x < n2; x += 32) m = fmax(m, l[x]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    for (int x = lane; x < n2; x += 32) {          // terms below e^-50 of the largest cannot change the rounded sum; NaN stays out
      const double v = l[x] - m;
      if (v > -50.0) s += exp(v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) lse[r] = s > 0.0 ? m + log(s) : -CUDART_INF;
  }
  __syncthreads();
  for (int x = threadIdx.x; x < gn; x += kThreads) {
    const int u = x / n2;
    const double L1 = rows[x] - lse[u], L2 = rows[gn + x] - lse[g + u];
    out[x] = L1 >= L2 ? L1 : L2;
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
int launch_logits(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* l_max, double* l_min, unsigned* done,
                  cudaStream_t st) {
  const dim3 grid(unsigned((m.n2 + kWarps - 1) / kWarps), unsigned(m.B * m.Hkv));
  const size_t smem = size_t(m.g) * m.d * m.es;    // the group's queries: up to 64 KB (fp32, 128 channels, 128 heads)
  if (smem > 30 * 1024 &&                          // 48 KB with the kernel's own
      cudaFuncSetAttribute(decode_logits_kernel<T, LPR>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
    return CP_ERR_CUDA;
  return launch_pdl(decode_logits_kernel<T, LPR>, grid, kThreads, smem, st, static_cast<const T*>(q_last),
                    static_cast<const char*>(K), p.k_stride[0], p.k_stride[1], p.k_stride[2], m.Hkv, m.g, m.n, m.blk, m.n2,
                    double(p.est_scale), l_max, l_min, done);
}

}  // namespace

// Blocks of up to 128 rows (a warp each), and query groups whose Kmin logits fit the workspace's key representatives
// ([B,Hkv,n2,d] twice), whose place they take: 8 g <= 2 d es, at least 32 heads per KV head.
bool decode_path_applies(const Dims& m) { return m.blk <= 128 && 8 * m.g <= 2 * m.d * m.es && m.B * (long long)m.Hkv <= 65535; }

int launch_decode_score(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* S_out, char* ws, cudaStream_t st) {
  double* l_min = reinterpret_cast<double*>(ws + ws_layout(m).kmax);
  unsigned* done = fused_rows(m) ? reinterpret_cast<unsigned*>(ws + sizeof(DeviceStatus)) : nullptr;
  const int lpr = m.d * m.es / 16;
  int rc = CP_ERR_UNSUPPORTED;
  if (p.dtype == CP_BF16)
    rc = lpr == 16 ? launch_logits<__nv_bfloat16, 16>(p, m, q_last, K, S_out, l_min, done, st) : launch_logits<__nv_bfloat16, 8>(p, m, q_last, K, S_out, l_min, done, st);
  else if (p.dtype == CP_F16)
    rc = lpr == 16 ? launch_logits<__half, 16>(p, m, q_last, K, S_out, l_min, done, st) : launch_logits<__half, 8>(p, m, q_last, K, S_out, l_min, done, st);
  else
    rc = lpr == 32 ? launch_logits<float, 32>(p, m, q_last, K, S_out, l_min, done, st) : launch_logits<float, 16>(p, m, q_last, K, S_out, l_min, done, st);
  if (rc != CP_OK || done != nullptr) return rc;
  const dim3 grid(unsigned(m.B * m.Hq));
  if (m.n2 <= 4 * kThreads) return launch_pdl(decode_score_kernel<4>, grid, kThreads, 0, st, S_out, l_min, m.n2);
  if (m.n2 <= 16 * kThreads) return launch_pdl(decode_score_kernel<16>, grid, kThreads, 0, st, S_out, l_min, m.n2);
  return launch_pdl(decode_score_kernel<32>, grid, kThreads, 0, st, S_out, l_min, m.n2);
}

}  // namespace cp
