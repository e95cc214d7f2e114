// Per-channel max / min over rows of 16-byte slices, shared by the kernels that read Q and K (Algorithm 1, lines 7-8).
#pragma once
#include "cp_common.cuh"

namespace cp {
namespace {

template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> {
  uint4 v;
  static constexpr uint32_t kNegInf = 0xFF80FF80u, kPosInf = 0x7F807F80u;   // packed pairs
  __device__ static Vec load(const void* p) { Vec r; r.v = __ldg(reinterpret_cast<const uint4*>(p)); return r; }
  __device__ void store(void* p) const { *reinterpret_cast<uint4*>(p) = v; }
  __device__ static uint32_t mx(uint32_t a, uint32_t b) {
    __nv_bfloat162 r = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<uint32_t*>(&r);
  }
  __device__ static uint32_t mn(uint32_t a, uint32_t b) {
    __nv_bfloat162 r = __hmin2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<uint32_t*>(&r);
  }
};
template <> struct Vec<__half> {
  uint4 v;
  static constexpr uint32_t kNegInf = 0xFC00FC00u, kPosInf = 0x7C007C00u;
  __device__ static Vec load(const void* p) { Vec r; r.v = __ldg(reinterpret_cast<const uint4*>(p)); return r; }
  __device__ void store(void* p) const { *reinterpret_cast<uint4*>(p) = v; }
  __device__ static uint32_t mx(uint32_t a, uint32_t b) {
    __half2 r = __hmax2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
    return *reinterpret_cast<uint32_t*>(&r);
  }
  __device__ static uint32_t mn(uint32_t a, uint32_t b) {
    __half2 r = __hmin2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
    return *reinterpret_cast<uint32_t*>(&r);
  }
};
template <> struct Vec<float> {
  uint4 v;
  static constexpr uint32_t kNegInf = 0xFF800000u, kPosInf = 0x7F800000u;
  __device__ static Vec load(const void* p) { Vec r; r.v = __ldg(reinterpret_cast<const uint4*>(p)); return r; }
  __device__ void store(void* p) const { *reinterpret_cast<uint4*>(p) = v; }
  __device__ static uint32_t mx(uint32_t a, uint32_t b) { return __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b))); }
  __device__ static uint32_t mn(uint32_t a, uint32_t b) { return __float_as_uint(fminf(__uint_as_float(a), __uint_as_float(b))); }
};

template <typename T>
__device__ __forceinline__ void vmax(uint4& a, const uint4& b) {
  a.x = Vec<T>::mx(a.x, b.x); a.y = Vec<T>::mx(a.y, b.y); a.z = Vec<T>::mx(a.z, b.z); a.w = Vec<T>::mx(a.w, b.w);
}
template <typename T>
__device__ __forceinline__ void vmin(uint4& a, const uint4& b) {
  a.x = Vec<T>::mn(a.x, b.x); a.y = Vec<T>::mn(a.y, b.y); a.z = Vec<T>::mn(a.z, b.z); a.w = Vec<T>::mn(a.w, b.w);
}
__device__ __forceinline__ uint4 shfl_xor4(const uint4& a, int m) {
  uint4 r;
  r.x = __shfl_xor_sync(0xffffffffu, a.x, m); r.y = __shfl_xor_sync(0xffffffffu, a.y, m);
  r.z = __shfl_xor_sync(0xffffffffu, a.z, m); r.w = __shfl_xor_sync(0xffffffffu, a.w, m);
  return r;
}

// Fold rows first+sub, first+sub+step, ... (< first+nrows) of a group into the lane's 16-byte
// slice of (max, min).  The accumulators start at -inf / +inf, so a lane without rows is neutral.
template <typename T, int LPR>
__device__ __forceinline__ void scan_rows(const char* gbase, int64_t st_bytes, int first, int nrows,
                                          int step, int lane, uint4& mx, uint4& mn) {
  const int sub = lane / LPR, col = lane % LPR;
  const char* p0 = gbase + int64_t(first + sub) * st_bytes + col * 16;
  mx = make_uint4(Vec<T>::kNegInf, Vec<T>::kNegInf, Vec<T>::kNegInf, Vec<T>::kNegInf);
  mn = make_uint4(Vec<T>::kPosInf, Vec<T>::kPosInf, Vec<T>::kPosInf, Vec<T>::kPosInf);
  constexpr int UNROLL = 8;
  int i = first + sub;
  const int end = first + nrows;
  for (; i + (UNROLL - 1) * step < end; i += UNROLL * step) {
    uint4 v[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) v[u] = Vec<T>::load(p0 + int64_t(i - first - sub + u * step) * st_bytes).v;
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) { vmax<T>(mx, v[u]); vmin<T>(mn, v[u]); }
  }
  for (; i < end; i += step) {
    const uint4 v = Vec<T>::load(p0 + int64_t(i - first - sub) * st_bytes).v;
    vmax<T>(mx, v); vmin<T>(mn, v);
  }
}

}  // namespace
}  // namespace cp
