// SIMT attention over a block list (Algorithm 2, lines 6-13) and dense causal attention (Eq. 2), fp32 arithmetic on the
// FMA pipes: the path for fp32 inputs and for shapes outside the tensor-core envelope (blocks or segments that are not
// multiples of its tiles).
//
// One CTA = BM query rows of one head and segment against key tiles of 64 tokens gathered from the block list.  128 threads
// = 16 key (channel) columns x 8 row groups; a thread holds an RT x 4 piece of S and an RT x D/16 piece of O, so 4 channels
// cost RT + 4 16-byte shared loads per 16 RT FMAs.  K, V tiles arrive by cp.async (the next K tile under softmax and P V,
// the V tile under Q K^T).  Bound by FMA issue and shared-memory loads (36 TFLOP/s at 3 x 4000 tokens x 8 heads x 64 channels,
// budget 4096).  A warp per row, which this replaced, read every key once per row: 1024 tokens x 4 heads x 64 channels, budget
// 256, fp32: 230 us, here 17 us; error against fp64 at or below that kernel's (9.22e-7 against 9.24e-7 relative at 4001 tokens).
#include <math_constants.h>

#include <algorithm>

#include "cp_common.cuh"

namespace cp {
namespace {

constexpr int kThreads = 128;    // of one key group
constexpr int kBN = 64;          // keys per tile

template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }
template <> __device__ __forceinline__ float to_f32<__half>(__half x) { return __half2float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ __half from_f32<__half>(float x) { return __float2half_rn(x); }
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// four consecutive elements of shared memory as fp32
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <typename T> __device__ __forceinline__ float4 ld4(const T* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  const T* e = reinterpret_cast<const T*>(&v);
  return make_float4(to_f32(e[0]), to_f32(e[1]), to_f32(e[2]), to_f32(e[3]));
}

// 16 bytes global -> shared, zeros when !valid (the source is then not read)
__device__ __forceinline__ void cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T>
struct SimtArgs {
  const T *Q, *K, *V;
  T* O;
  const int32_t *idx, *cnt;
  float* lse;
  DeviceStatus* st;
  int B, Hq, g, n, seg, blk, k, r, dense, tiles_per_seg;
  int64_t qs[3], ks[3], vs[3], os[3];
  float sm_scale;
};

// One row by one warp over exactly the keys it sees, in fp32.  In a tile a key that a row does not see enters that row's sum
// with probability zero, which is NaN where the key's value is infinite or NaN; rows that came out so are done again here.
template <typename T, int D>
__device__ __noinline__ void exact_row(const SimtArgs<T>* ap, int b, int h, int t, const int32_t* list, int n_ranges, int lane) {
  const SimtArgs<T>& a = *ap;
  const T* q = a.Q + b * a.qs[0] + h * a.qs[1] + int64_t(t) * a.qs[2];
  const T* Kh = a.K + b * a.ks[0] + (h / a.g) * a.ks[1];
  const T* Vh = a.V + b * a.vs[0] + (h / a.g) * a.vs[1];
  constexpr int CPL = D / 32;   // output channels per lane
  float acc[CPL];
#pragma unroll
  for (int i = 0; i < CPL; ++i) acc[i] = 0.f;
  float m_run = -CUDART_INF_F, l_run = 0.f;
  for (int e = 0; e < n_ranges; ++e) {
    const int u0 = a.dense ? 0 : list[e] * a.blk, u1 = a.dense ? t + 1 : min(u0 + a.blk, t + 1);
    for (int base = u0; base < u1; base += 32) {
      const int u = base + lane;
      float s = -CUDART_INF_F;
      if (u < u1) {
        const T* kr = Kh + int64_t(u) * a.ks[2];
        float x = 0.f;
        for (int c = 0; c < D; ++c) x = fmaf(to_f32(q[c]), to_f32(kr[c]), x);
        s = x * a.sm_scale;
      }
      float mx = s;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(m_run, mx);
      const float corr = (m_run == -CUDART_INF_F) ? 0.f : expf(m_run - m_new);
      const float p = (u < u1) ? expf(s - m_new) : 0.f;
      float ps = p;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
      l_run = l_run * corr + ps;
      m_run = m_new;
#pragma unroll
      for (int i = 0; i < CPL; ++i) acc[i] *= corr;
      const int here = min(32, u1 - base);
      for (int kk = 0; kk < here; ++kk) {
        const float pk = __shfl_sync(0xffffffffu, p, kk);
        const T* vr = Vh + int64_t(base + kk) * a.vs[2];
#pragma unroll
        for (int i = 0; i < CPL; ++i) acc[i] = fmaf(pk, to_f32(vr[lane + 32 * i]), acc[i]);
      }
    }
  }
  T* o = a.O + b * a.os[0] + h * a.os[1] + int64_t(t) * a.os[2];
  const float inv = l_run > 0.f ? 1.f / l_run : 0.f;   // a row without any visible key: zeros, lse = ln 0
#pragma unroll
  for (int i = 0; i < CPL; ++i) o[lane + 32 * i] = from_f32<T>(acc[i] * inv);
  if (a.lse != nullptr && lane == 0) a.lse[((long long)b * a.Hq + h) * a.n + t] = m_run + logf(l_run);
}

template <typename T, int D, int RT, int NG>
struct SimtShape {
  static constexpr int kBM = RT * (kThreads / 16);
  static constexpr int kKS = D + 16 / int(sizeof(T));   // row stride of a K / V tile: 16 bytes of padding
  static constexpr int kPS = kBN + 4;
  static constexpr size_t kGroup = 2 * size_t(kBN) * kKS * sizeof(T) + size_t(kBM) * kPS * 4;   // K, V and P of a group
  static constexpr size_t kSmem = size_t(kBM) * (D + 4) * 4 + NG * kGroup;
  static_assert(kThreads * RT * (D / 16 + 2) * 4 <= kGroup, "a group leaves its partial result where its tiles were");
};

// NG groups of 128 threads walk the key tiles of the same rows, every NG-th tile each, and merge their (O, max, sum) at the end.
template <typename T, int D, int RT, int NG>
__global__ void __launch_bounds__(kThreads * NG)
attention_simt_kernel(const __grid_constant__ SimtArgs<T> a) {
  using S = SimtShape<T, D, RT, NG>;
  constexpr int kBM = S::kBM, kKS = S::kKS, kPS = S::kPS, kQS = D + 4;
  const int32_t* idx = a.idx;
  pdl_trigger();
  pdl_wait(idx);
  extern __shared__ __align__(16) uint8_t smem[];
  float* qs = reinterpret_cast<float*>(smem);              // [kBM][kQS]
  const int grp = NG > 1 ? threadIdx.x / kThreads : 0;
  float* ps = qs + kBM * kQS + grp * int(S::kGroup / 4);    // [kBM][kPS]
  T* kt = reinterpret_cast<T*>(ps + kBM * kPS);             // [kBN][kKS]
  T* vt = kt + kBN * kKS;
  __shared__ int tok_all[NG][2][kBN];                         // token of each key of the tile; 0x7fffffff: no such key
  __shared__ int list_state[2];                             // [0] the list is valid, [1] listed keys up to the last row
  __shared__ int redo[kBM];

  const int tid = threadIdx.x % kThreads, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int (*tok_sh)[kBN] = tok_all[grp];
  auto group_sync = [&] {
    if constexpr (NG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kThreads) : "memory");
  };
  const int tx = tid & 15, ty = tid >> 4;
  // CTA -> (row tile, batch * head): heads fastest, the latest tiles (most keys) first
  const int BH = a.B * a.Hq;
  const int bh = blockIdx.x % BH;
  const int tile = int(gridDim.x / BH) - 1 - int(blockIdx.x) / BH;
  const int h = bh % a.Hq, b = bh / a.Hq;
  const int j = tile / a.tiles_per_seg;
  const int t0 = j * a.seg + (tile % a.tiles_per_seg) * kBM;
  const int t_end = min(min(t0 + kBM, (j + 1) * a.seg), a.n);      // rows [t0, t_end)
  if (t0 >= t_end) return;
  const int n1 = (a.n + a.seg - 1) / a.seg, n2 = (a.n + a.blk - 1) / a.blk;

  // Everything the first tile needs is asked for at once: the list and its length, the tokens of the tile's keys, the rows of Q.  One after
  // the other -- length, list, rows, tokens -- it was three to four round trips: whole layer, 1024 tokens x 4 heads x 64 channels, fp32, caches
  // cold, 30.9 us, now 29.6 (a third of the attention's 16.5 us is such latency).
  const int32_t* list = nullptr;
  int cnt = 0, n_keys = t_end;                                      // positions of the key sequence the CTA walks
  if (!a.dense) {
    const long long u = (long long)bh * n1 + j;
    list = idx + u * a.k;
    cnt = a.cnt[u];
  }
  // token of a position, 0x7fffffff: none.  An entry that is no block of the sequence is not followed, whatever the list turns out to be.
  auto token_at = [&](int pos) {
    if (a.dense) return pos < t_end ? pos : 0x7fffffff;
    const int e = pos / a.blk;
    const int entry = e < a.k ? __ldg(list + e) : -1;
    if (e >= cnt || uint32_t(entry) >= uint32_t(n2)) return 0x7fffffff;
    const int tok = entry * a.blk + pos % a.blk;
    return tok < t_end ? tok : 0x7fffffff;
  };
  auto make_tokens = [&](int tile_i) {                               // threads 0..63
    if (tid < kBN) tok_sh[(tile_i / NG) & 1][tid] = token_at(tile_i * kBN + tid);
  };
  // Q rows, widened to fp32
  const T* qg = a.Q + b * a.qs[0] + h * a.qs[1];
  for (int e = threadIdx.x; e < kBM * (D / 4); e += kThreads * NG) {
    const int row = e / (D / 4), c4 = e % (D / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + row < t_end) v = ld4(qg + int64_t(t0 + row) * a.qs[2] + c4 * 4);
    *reinterpret_cast<float4*>(qs + row * kQS + c4 * 4) = v;
  }
  make_tokens(grp);
  for (int i = threadIdx.x; i < kBM; i += kThreads * NG) redo[i] = 0;
  if (!a.dense) {
    if (warp == 0) {
      bool ok = cnt >= 0 && cnt <= a.k;
      const int vis = min(n2, (j + 1) * a.r);
      int end = 0;                                                  // positions up to the last key that a row can see
      for (int i = lane; i < a.k; i += 32) {
        const int v = list[i], before = i > 0 ? list[i - 1] : -1;
        if (i < cnt) {
          ok = ok && v >= 0 && v < vis && before < v;
          if (v * a.blk < t_end) end = max(end, i * a.blk + min(a.blk, t_end - v * a.blk));
        }
      }
      ok = __all_sync(0xffffffffu, ok);
      // the list is ascending: later blocks are seen by no row, and of the last one only the keys up to the last row
      end = __reduce_max_sync(0xffffffffu, end);
      if (lane == 0) { list_state[0] = ok; list_state[1] = end; }
    }
    __syncthreads();
    if (!list_state[0]) {
      if (threadIdx.x == 0 && t0 == j * a.seg) report(a.st, CP_ERR_BOUNDS, 100, b, h, j, cnt);
      return;
    }
    n_keys = list_state[1];
  } else {
    __syncthreads();
  }

  const T* kg = a.K + b * a.ks[0] + (h / a.g) * a.ks[1];
  const T* vg = a.V + b * a.vs[0] + (h / a.g) * a.vs[1];
  const int n_tiles = (n_keys + kBN - 1) / kBN;
  constexpr int VPR = D * int(sizeof(T)) / 16;                        // 16-byte vectors per row
  auto load_tile = [&](const T* base, int64_t stride, T* dst, int tile_i) {
    for (int e = tid; e < kBN * VPR; e += kThreads) {
      const int key = e / VPR, c = e % VPR;
      const int tok = tok_sh[(tile_i / NG) & 1][key];
      const bool valid = tok != 0x7fffffff;
      cp16(dst + key * kKS + c * (16 / int(sizeof(T))), base + int64_t(valid ? tok : 0) * stride + c * (16 / int(sizeof(T))), valid);
    }
    cp_commit();
  };

  float o[RT][D / 16], m_run[RT], l_run[RT];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    m_run[i] = -CUDART_INF_F; l_run[i] = 0.f;
#pragma unroll
    for (int c = 0; c < D / 16; ++c) o[i][c] = 0.f;
  }
  if (grp < n_tiles) load_tile(kg, a.ks[2], kt, grp);
  for (int it = grp; it < n_tiles; it += NG) {
    load_tile(vg, a.vs[2], vt, it);                                   // lands under Q K^T
    if (it + NG < n_tiles) make_tokens(it + NG);
    cp_wait<1>();                                                     // the K tile
    group_sync();  

    // S = Q K^T: rows ty*RT + i, keys tx + 16 jj
    float s[RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) s[i][jj] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      float4 kv[4];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) kv[jj] = ld4(kt + (tx + 16 * jj) * kKS + c);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float4 qv = ld4(qs + (ty * RT + i) * kQS + c);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          s[i][jj] = fmaf(qv.x, kv[jj].x, s[i][jj]);
          s[i][jj] = fmaf(qv.y, kv[jj].y, s[i][jj]);
          s[i][jj] = fmaf(qv.z, kv[jj].z, s[i][jj]);
          s[i][jj] = fmaf(qv.w, kv[jj].w, s[i][jj]);
        }
      }
    }
    // mask, online softmax (the 16 threads of a row group are 16 neighbouring lanes), P to shared memory
    int tok[4];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) tok[jj] = tok_sh[(it / NG) & 1][tx + 16 * jj];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int t = t0 + ty * RT + i;
      float mx = -CUDART_INF_F;
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        s[i][jj] = tok[jj] <= t ? s[i][jj] * a.sm_scale : -CUDART_INF_F;
        mx = fmaxf(mx, s[i][jj]);
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
      const float m_new = fmaxf(m_run[i], mx);
      const float m_ref = m_new == -CUDART_INF_F ? 0.f : m_new;       // no visible key so far: every p is exp(-inf) = 0
      const float corr = m_run[i] == -CUDART_INF_F ? 0.f : expf(m_run[i] - m_new);
      m_run[i] = m_new;
      float sum = 0.f;
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const float p = expf(s[i][jj] - m_ref);
        ps[(ty * RT + i) * kPS + tx + 16 * jj] = p;
        sum += p;
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
      l_run[i] = l_run[i] * corr + sum;
#pragma unroll
      for (int c = 0; c < D / 16; ++c) o[i][c] *= corr;
    }
    group_sync();                                                    // the K tile has been read, tokens of the next tile are there
    if (it + NG < n_tiles) { load_tile(kg, a.ks[2], kt, it + NG); cp_wait<1>(); }
    else cp_wait<0>();
    group_sync();                                                    // the V tile

    // O += P V: channels tx*4 + 64 q
#pragma unroll 2
    for (int kk = 0; kk < kBN; kk += 4) {
      float4 pv[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) pv[i] = ld4(ps + (ty * RT + i) * kPS + kk);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
#pragma unroll
        for (int q = 0; q < D / 64; ++q) {
          const float4 v = ld4(vt + (kk + x) * kKS + q * 64 + tx * 4);
#pragma unroll
          for (int i = 0; i < RT; ++i) {
            const float p = x == 0 ? pv[i].x : (x == 1 ? pv[i].y : (x == 2 ? pv[i].z : pv[i].w));
            o[i][q * 4 + 0] = fmaf(p, v.x, o[i][q * 4 + 0]);
            o[i][q * 4 + 1] = fmaf(p, v.y, o[i][q * 4 + 1]);
            o[i][q * 4 + 2] = fmaf(p, v.z, o[i][q * 4 + 2]);
            o[i][q * 4 + 3] = fmaf(p, v.w, o[i][q * 4 + 3]);
          }
        }
      }
    }
    group_sync();                                                    // V and P have been read
  }

  if constexpr (NG > 1) {
    // groups 1.. leave (O, max, sum) where their tiles were; group 0 merges them into its own
    constexpr int OC = D / 16;
    float* mine = qs + kBM * kQS + grp * int(S::kGroup / 4);
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < RT; ++i) {
#pragma unroll
        for (int c = 0; c < OC; ++c) mine[(i * (OC + 2) + c) * kThreads + tid] = o[i][c];
        mine[(i * (OC + 2) + OC) * kThreads + tid] = m_run[i];
        mine[(i * (OC + 2) + OC + 1) * kThreads + tid] = l_run[i];
      }
    }
    __syncthreads();
    if (grp == 0) {
#pragma unroll 1
      for (int g2 = 1; g2 < min(NG, n_tiles); ++g2) {
        const float* other = qs + kBM * kQS + g2 * int(S::kGroup / 4);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float m2 = other[(i * (OC + 2) + OC) * kThreads + tid], l2 = other[(i * (OC + 2) + OC + 1) * kThreads + tid];
          const float m_new = fmaxf(m_run[i], m2);
          const float f1 = m_run[i] == -CUDART_INF_F ? 0.f : expf(m_run[i] - m_new), f2 = m2 == -CUDART_INF_F ? 0.f : expf(m2 - m_new);
          m_run[i] = m_new;
          l_run[i] = l_run[i] * f1 + l2 * f2;
#pragma unroll
          for (int c = 0; c < OC; ++c) o[i][c] = o[i][c] * f1 + other[(i * (OC + 2) + c) * kThreads + tid] * f2;
        }
      }
    }
  }

  T* og = a.O + b * a.os[0] + h * a.os[1];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int row = ty * RT + i, t = t0 + row;
    if (t >= t_end || (NG > 1 && grp > 0)) continue;
    const float inv = l_run[i] > 0.f ? 1.f / l_run[i] : 0.f;         // a row without any visible key: zeros, lse = ln 0
    float odd = l_run[i] > 0.f ? 0.f : CUDART_NAN_F;
#pragma unroll
    for (int q = 0; q < D / 64; ++q) {
      T w[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) { w[c] = from_f32<T>(o[i][q * 4 + c] * inv); odd = fmaf(o[i][q * 4 + c], 0.f, odd); }
      T* dst = og + int64_t(t) * a.os[2] + q * 64 + tx * 4;
      if constexpr (sizeof(T) == 4) *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(w);
      else *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(w);
    }
    if (!(odd == 0.f)) redo[row] = 1;
    if (a.lse != nullptr && tx == 0) a.lse[(long long)bh * a.n + t] = m_run[i] + logf(l_run[i]);
  }
  __syncthreads();
  for (int row = warp; row < t_end - t0; row += kThreads * NG / 32)
    if (redo[row]) exact_row<T, D>(&a, b, h, t0 + row, list, a.dense ? 1 : cnt, lane);
}

template <typename T, int D, int RT, int NG>
int launch_rt(const SimtArgs<T>& a0, const Dims& m, cudaStream_t s) {
  using S = SimtShape<T, D, RT, NG>;
  SimtArgs<T> a = a0;
  // no segment has more rows than the sequence; the last one may be shorter than that: its missing tiles return at once
  a.tiles_per_seg = (std::min(m.seg, m.n) + S::kBM - 1) / S::kBM;
  const long long ctas = (long long)m.B * m.Hq * m.n1 * a.tiles_per_seg;
  if (ctas > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  auto kern = attention_simt_kernel<T, D, RT, NG>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(S::kSmem)) != cudaSuccess) return CP_ERR_CUDA;
  return launch_pdl(kern, dim3(unsigned(ctas)), kThreads * NG, S::kSmem, s, a);
}

template <typename T, int D>
int launch_t(const cp_params& p, const Dims& m, const void* Q, const void* K, const void* V,
             const int32_t* idx, const int32_t* cnt, void* O, float* lse, DeviceStatus* st, bool dense,
             cudaStream_t s) {
  SimtArgs<T> a;
  a.Q = static_cast<const T*>(Q); a.K = static_cast<const T*>(K); a.V = static_cast<const T*>(V); a.O = static_cast<T*>(O);
  a.idx = idx; a.cnt = cnt; a.lse = lse; a.st = st;
  a.B = m.B; a.Hq = m.Hq; a.g = m.g; a.n = m.n; a.seg = m.seg; a.blk = m.blk; a.k = m.k; a.r = m.r; a.dense = dense ? 1 : 0;
  for (int i = 0; i < 3; ++i) { a.qs[i] = p.q_stride[i]; a.ks[i] = p.k_stride[i]; a.vs[i] = p.v_stride[i]; a.os[i] = p.o_stride[i]; }
  a.sm_scale = p.sm_scale;
  // Up to four CTAs of 32 rows per SM a CTA's tiles are spread over key groups (as many as shared memory holds), which shortens
  // the chain of tiles a small problem waits for: 1500 tokens x 4 heads x 64 channels 79 -> 51 us, 2047 x 8 x 128: 261 -> 236,
  // even at 2047 x 8 x 64 (131 us).  Beyond that throughput counts: 64 channels take 64 rows per CTA (4000 x 8, budget 2048:
  // 358 us against 438 with 32 rows and 431 in groups), 128 channels 32 rows in one group, so that two CTAs fit an SM (766 us
  // against 867 and 817).
  constexpr int kNG = D * sizeof(T) <= 256 ? 4 : 2;
  const long long ctas32 = (long long)m.B * m.Hq * ((m.n + 31) / 32);
  if (ctas32 < 4 * 148) return launch_rt<T, D, 4, kNG>(a, m, s);
  if constexpr (D == 64)
    if (m.seg >= 64) return launch_rt<T, D, 8, 1>(a, m, s);
  return launch_rt<T, D, 4, 1>(a, m, s);
}

}  // namespace

int launch_attention_simt(const cp_params& p, const Dims& m, const void* Q, const void* K,
                          const void* V, const int32_t* idx, const int32_t* cnt, void* O, float* lse,
                          DeviceStatus* st, bool dense, cudaStream_t s) {
  if (p.dtype == CP_BF16) {
    if (m.d == 128) return launch_t<__nv_bfloat16, 128>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
    if (m.d == 64) return launch_t<__nv_bfloat16, 64>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
  } else if (p.dtype == CP_F16) {
    if (m.d == 128) return launch_t<__half, 128>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
    if (m.d == 64) return launch_t<__half, 64>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
  } else {
    if (m.d == 128) return launch_t<float, 128>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
    if (m.d == 64) return launch_t<float, 64>(p, m, Q, K, V, idx, cnt, O, lse, st, dense, s);
  }
  return CP_ERR_UNSUPPORTED;
}

}  // namespace cp
