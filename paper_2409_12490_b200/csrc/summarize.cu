// K1: per-channel max / min over the tokens of each query segment and each key block
// (Algorithm 1, lines 3-8).  Pure HBM scan: 16-byte loads, comparisons only, results exact
// in the input dtype.
//
// One launch covers Q (groups of `seg` rows) and K (groups of `blk` rows).  A row of d
// elements is read by LPR = d*es/16 neighbouring lanes, so a warp covers 32/LPR rows per
// load instruction.  Groups of <= 128 rows are owned by one warp; larger groups by a whole
// CTA whose warps stride over the rows and combine through shared memory.
#include "summarize.cuh"

namespace cp {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;

// largest magnitude among the elements of a 16-byte vector
template <typename T> __device__ __forceinline__ float vec_absmax(const uint4& a);
template <> __device__ __forceinline__ float vec_absmax<float>(const uint4& a) {
  return fmaxf(fmaxf(fabsf(__uint_as_float(a.x)), fabsf(__uint_as_float(a.y))), fmaxf(fabsf(__uint_as_float(a.z)), fabsf(__uint_as_float(a.w))));
}
template <> __device__ __forceinline__ float vec_absmax<__nv_bfloat16>(const uint4& a) {
  const uint32_t w[4] = {a.x, a.y, a.z, a.w};
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {   // a bf16 is the upper half of a float
    m = fmaxf(m, fabsf(__uint_as_float(w[i] << 16)));
    m = fmaxf(m, fabsf(__uint_as_float(w[i] & 0xffff0000u)));
  }
  return m;
}
template <> __device__ __forceinline__ float vec_absmax<__half>(const uint4& a) {
  const uint32_t w[4] = {a.x, a.y, a.z, a.w};
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
    m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
  }
  return m;
}
// largest magnitude of a group's summaries: every lane holds the group's (max, min) slice of column slot lane % LPR
template <typename T, int LPR>
__device__ __forceinline__ float group_absmax(const uint4& mx, const uint4& mn) {
  float m = fmaxf(vec_absmax<T>(mx), vec_absmax<T>(mn));
#pragma unroll
  for (int o = 1; o < LPR; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m;
}

struct Side {            // one tensor (Q or K) and where its summaries go
  const char* base;      // element (b,h,t,0) at base + (b*sb + h*sh + t*st) * es
  int64_t sb, sh, st;    // strides in elements
  int H, groups_per_head, G, n;  // heads, groups per head (ceil(n/G)), rows per group (the last may be shorter), tokens
  char *omax, *omin;     // [B,H,groups,d] contiguous
  float* oabs;           // nullable, [B,H,groups]: largest magnitude in the group's summaries
  long long n_groups;    // B*H*groups_per_head
  long long cta_begin;   // first CTA of this side
  int groups_per_cta;    // kWarps (warp-owned groups) or 1 (CTA-owned group)
};

template <int NS> struct Sides { Side s[2 * NS]; int n; };   // Q and K of each sequence, by cta_begin

template <typename T, int LPR, int NS>
__global__ void __launch_bounds__(kThreads) summarize_kernel(const __grid_constant__ Sides<NS> t, int d) {
  __shared__ uint4 red[2][kWarps][LPR];
  int si = 0;
  while (si + 1 < t.n && blockIdx.x >= t.s[si + 1].cta_begin) ++si;
  const Side& s = t.s[si];
  const char* base = s.base;
  pdl_trigger();
  pdl_wait(base);
  const long long cta = blockIdx.x - s.cta_begin;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int RPW = 32 / LPR;
  const int es = sizeof(T);
  const int64_t st_bytes = s.st * es;

  if (s.groups_per_cta == 1) {
    // a CTA owns the group; its warps take rows warp*RPW + sub, stride kWarps*RPW
    const long long grp = cta;
    const int gi = int(grp % s.groups_per_head);
    const long long bh = grp / s.groups_per_head;
    const int h = int(bh % s.H), b = int(bh / s.H);
    const char* gbase = base + (int64_t(b) * s.sb + int64_t(h) * s.sh + int64_t(gi) * s.G * s.st) * es;
    const int rows = min(s.G, s.n - gi * s.G);
    uint4 mx, mn;
    scan_rows<T, LPR>(gbase, st_bytes, warp * RPW, rows - warp * RPW, kWarps * RPW, lane, mx, mn);
#pragma unroll
    for (int m = LPR; m < 32; m <<= 1) { uint4 o = shfl_xor4(mx, m); vmax<T>(mx, o); o = shfl_xor4(mn, m); vmin<T>(mn, o); }
    if (lane < LPR) { red[0][warp][lane] = mx; red[1][warp][lane] = mn; }
    __syncthreads();
    if (warp == 0) {
      const int col = lane % LPR;
      mx = red[0][0][col]; mn = red[1][0][col];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) { vmax<T>(mx, red[0][w][col]); vmin<T>(mn, red[1][w][col]); }
      if (lane < LPR) {
        const size_t off = (size_t(grp) * d) * es + lane * 16;
        *reinterpret_cast<uint4*>(s.omax + off) = mx;
        *reinterpret_cast<uint4*>(s.omin + off) = mn;
      }
      if (s.oabs != nullptr) {
        const float am = group_absmax<T, LPR>(mx, mn);
        if (lane == 0) s.oabs[grp] = am;
      }
    }
  } else {
    // each warp owns one group of G <= 128 rows
    const long long grp = cta * kWarps + warp;
    if (grp >= s.n_groups) return;
    const int gi = int(grp % s.groups_per_head);
    const long long bh = grp / s.groups_per_head;
    const int h = int(bh % s.H), b = int(bh / s.H);
    const char* gbase = base + (int64_t(b) * s.sb + int64_t(h) * s.sh + int64_t(gi) * s.G * s.st) * es;
    const int rows = min(s.G, s.n - gi * s.G);
    uint4 mx, mn;
    scan_rows<T, LPR>(gbase, st_bytes, 0, rows, RPW, lane, mx, mn);
#pragma unroll
    for (int m = LPR; m < 32; m <<= 1) { uint4 o = shfl_xor4(mx, m); vmax<T>(mx, o); o = shfl_xor4(mn, m); vmin<T>(mn, o); }
    if (lane < LPR) {
      const size_t off = (size_t(grp) * d) * es + lane * 16;
      *reinterpret_cast<uint4*>(s.omax + off) = mx;
      *reinterpret_cast<uint4*>(s.omin + off) = mn;
    }
    if (s.oabs != nullptr) {
      const float am = group_absmax<T, LPR>(mx, mn);
      if (lane == 0) s.oabs[grp] = am;
    }
  }
}

template <int NS>
int launch_sides(const cp_params& p, const Dims& m, const Sides<NS>& t, long long ctas, cudaStream_t st) {
  if (ctas > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  const dim3 grid(static_cast<unsigned>(ctas));
  const int lpr = m.d * m.es / 16;
  if (p.dtype == CP_BF16) {
    if (lpr == 16) return launch_pdl(summarize_kernel<__nv_bfloat16, 16, NS>, grid, kThreads, 0, st, t, m.d);
    if (lpr == 8) return launch_pdl(summarize_kernel<__nv_bfloat16, 8, NS>, grid, kThreads, 0, st, t, m.d);
  } else if (p.dtype == CP_F16) {
    if (lpr == 16) return launch_pdl(summarize_kernel<__half, 16, NS>, grid, kThreads, 0, st, t, m.d);
    if (lpr == 8) return launch_pdl(summarize_kernel<__half, 8, NS>, grid, kThreads, 0, st, t, m.d);
  } else {
    if (lpr == 32) return launch_pdl(summarize_kernel<float, 32, NS>, grid, kThreads, 0, st, t, m.d);
    if (lpr == 16) return launch_pdl(summarize_kernel<float, 16, NS>, grid, kThreads, 0, st, t, m.d);
  }
  return CP_ERR_UNSUPPORTED;
}

// appends the sides of one problem whose first token is `tok`; Q == nullptr: key side only (the caller supplies the query
// representatives itself)
template <int NS>
void add_problem(Sides<NS>& t, long long& ctas, const cp_params& p, const Dims& m, int64_t tok, const void* Q, const void* K, char* ws) {
  const WsLayout w = ws_layout(m);
  auto add = [&](const void* base, const int64_t* s, int H, int G, char* omax, char* omin, float* oabs) {
    Side& x = t.s[t.n++];
    x.base = static_cast<const char*>(base) + tok * s[2] * m.es; x.sb = s[0]; x.sh = s[1]; x.st = s[2];
    x.H = H; x.G = G; x.n = m.n; x.groups_per_head = (m.n + G - 1) / G; x.omax = omax; x.omin = omin; x.oabs = oabs;
    x.n_groups = (long long)m.B * H * x.groups_per_head;
    x.groups_per_cta = G > 128 ? 1 : kWarps;
    x.cta_begin = ctas;
    ctas += (x.n_groups + x.groups_per_cta - 1) / x.groups_per_cta;
  };
  if (Q != nullptr) add(Q, p.q_stride, m.Hq, m.seg, ws + w.qmax, ws + w.qmin, nullptr);
  add(K, p.k_stride, m.Hkv, m.blk, ws + w.kmax, ws + w.kmin, reinterpret_cast<float*>(ws + w.kabs));
}

}  // namespace

int launch_summarize(const cp_params& p, const Dims& m, const void* Q, const void* K, char* ws,
                     cudaStream_t st) {
  Sides<1> t;
  t.n = 0;
  long long ctas = 0;
  add_problem(t, ctas, p, m, 0, Q, K, ws);
  return launch_sides<1>(p, m, t, ctas, st);
}

int launch_summarize_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, char* const* ws, int n_seqs, const void* Q,
                          const void* K, cudaStream_t st) {
  for (int i = 0; i < n_seqs; i += kSeqsPerLaunch) {
    Sides<kSeqsPerLaunch> t;
    t.n = 0;
    long long ctas = 0;
    for (int x = i; x < n_seqs && x < i + kSeqsPerLaunch; ++x) add_problem(t, ctas, p, seq_dims(m, slots[x].len), slots[x].tok, Q, K, ws[x]);
    const int rc = launch_sides<kSeqsPerLaunch>(p, m, t, ctas, st);
    if (rc != CP_OK) return rc;
  }
  return CP_OK;
}

}  // namespace cp
