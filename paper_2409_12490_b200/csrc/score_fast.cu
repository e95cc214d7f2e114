// K2 for 16-bit inputs with head_dim 128 (Algorithm 1, lines 9-14), split in two kernels:
//   lse (lse_sm100.cu)   the four log-sum-exps of every (head, segment) row, which need every key block of the row but only to
//        the accuracy with which a term can still change the sum, and
//   score_visible_kernel (this file)   the exact logits of the blocks a segment can see, combined straight out of tensor memory:
//        ln S = max( ln((S1+S3)/2), ln((S2+S4)/2) ), fusion with S'.
// Blocks that start at or after the end of the segment are masked by line 13 whatever their logits, so exact products are
// spent on the visible half of the map only.
//
// Exact products without the fp64 pipe.  A representative is an integer multiple of a power of two: with 2^E above the largest
// magnitude of its row, X = v 2^(30-E) is an integer of 31 bits unless v is smaller than the row's largest by some 2^22, and X is the
// sum of four signed bytes, d0 + d1 2^8 + d2 2^16 + d3 2^24.  A logit is then the sum of 16 products of byte rows, which
// tcgen05.mma.kind::i8 forms without any rounding; those of equal weight (i + j) share one of 7 accumulators of 32 bits (at most
// 2^23).  Put together in 64-bit integers and rounded once to fp64 they give the dot product correctly rounded, which a chain of 128
// fp64 additions does not.  Rows and blocks that do not fit (tiny values beside large ones, infinities, NaN) are marked, and their
// scores follow once more, from fp64 MMAs, at the end of their row group (redo_marked).
// What marks cost depends on the data.  Both kernels of the scores, us, 131072 tokens, 32 / 8 heads, segment 512, block 32, fused, fp16 with a
// channel of 80: 1 % of the blocks marked 608, 5 % 642, a third 929, all 1347 (840 with the products of all blocks on the fp64 pipe, whatever the
// values).  Normal bf16 inputs of that size have one marked row of 16384: 653 against 622 without.  With the marked logits summed by
// the threads that own them 1237, 1521, 3379, 7293 and 777.
//
// One CTA per SM, 128 logit rows (the Qmax / Qmin representatives of 64 / U segments x U heads of a KV group) against tiles
// of 32 key blocks (64 rows: Kmax, Kmin).  The tiles of all (row group, visible block) pairs are dealt to the CTAs in equal
// consecutive parts.  Roles (768 threads):
//   warps 0-15  epilogue: a thread per logit row and quarter of a tile; 7 accumulators -> logits, then the four logits of a score
//               meet in one of the two lanes that hold them (Qmax and Qmin rows alternate) and are combined in fp64; at the
//               start of a row group, the bytes of its query rows
//   warps 16-19 bytes of the next tile's key rows into shared memory
//   warp 20     MMA issuer: 64 MMAs of 128 x 64 x 32 per tile, under the fp64 part of the epilogue
//   warps 21-23 the masked part of the map: -inf
// No single unit bounds it (131072 tokens, segment 512, block 32; a tile takes some 10 thousand cycles): the byte MMAs and the fp64 operations hold the one
// pipe that they share 40 % of the cycles (their sum: they take turns), the data stage of shared memory is busy 56 % (MMA operands, 6 KB each, 31 %), few
// warps wait for it; they wait for tensor memory and for the fp64 pipe.  A tile's combination takes 1900 cycles alone (50 fp64 operations
// per score) and 6100 with the next tile's MMAs under way, which take 3400 to 4600.  8 epilogue warps: 14 thousand cycles per tile
// (latency).  Half tiles with accumulators of their own, so that half of the warps combine while the others convert: slower (N = 32: 5 KB per MMA of
// half the work; 131072 tokens 665 -> 780 us).
// Both kernels of the scores, this one with fp64 MMAs (m16n8k16, 8 to 12 warps each on its own tiles) -> now, us, in graphs, 32 / 8 heads:
// 131072 tokens, segment 512, block 32, fused, fp16 960 -> 622; segment 1024, block 128 193 -> 151.
#include "sm100_ptx.cuh"

namespace cp {
namespace {

constexpr int kEpilogueWarps = 16, kThreads = (kEpilogueWarps + 8) * 32, kMmaWarp = kEpilogueWarps + 4;
constexpr int kD = 128;
constexpr int kRows = 128;                     // logit rows (MMA M) per CTA
constexpr int kTileBlocks = 32;                // key blocks per tile
constexpr int kTileN = 2 * kTileBlocks;        // their Kmax rows, then their Kmin rows (MMA N)
constexpr int kDigits = 4, kAccs = 7;
constexpr int kQPlane = kRows * kD, kKPlane = kTileN * kD;      // bytes of one byte plane
constexpr int kStages = 2;                     // tiles of key rows
constexpr int kInfo = 4;                       // what goes with a tile (scales, marks) outlives its bytes: read until its epilogue ends
constexpr int kSmemK = kDigits * kQPlane;
constexpr int kSmemFixed = kSmemK + kStages * kDigits * kKPlane;
constexpr int kMarks = 512;                    // tiles whose marks are kept: a row group has at most kMaxBlocksN2 / kTileBlocks = 256, the converter is at most 2 ahead
static_assert(kMaxBlocksN2 / kTileBlocks + kStages <= kMarks, "marks of a row group");

constexpr int kNodes = 40 * 32 + 1;
static __device__ const double2 kSoftplusNodes[kNodes] = {
#include "softplus_nodes.inc"
};

struct Info {
  double scale[kTileBlocks];                   // 2^(E-30) of a block's bytes
};
struct __align__(16) RowInfo {
  double scale[kRows];                         // likewise for the logit rows
  double lse[kRows][2];                        // their log-sum-exps (Kmax, Kmin)
  uint8_t bad[kRows / 8], special[kRows / 8];  // marked rows, 8 per converting warp; whether some of the 8 have log-sum-exps that are not finite
};
struct Bars {
  double2 nodes[kNodes];                       // ln(1 + e^-x) and its derivative at the multiples of 1/32
  Info info[kInfo];
  RowInfo rows[2];                             // by parity of the CTA's row groups
  uint32_t marks[kMarks];                      // marked blocks of a tile, by the CTA's tiles
  uint16_t redo_blocks[kMaxBlocksN2];          // of a row group that has marks: its marked blocks, from its first on
  uint8_t redo_pairs[kRows / 2];               // and its marked (Qmax, Qmin) pairs of rows
  unsigned long long q_full, k_full[kStages], k_empty[kStages], info_full[kInfo], acc_full, acc_empty, redo;
  uint32_t tmem_base;
  volatile int abort_flag;
};
constexpr int kEpilogueRegs = 96, kOtherRegs = 48, kRegPoolNeeded = kEpilogueWarps * 32 * kEpilogueRegs + 256 * kOtherRegs;
constexpr int kSmemTotal = kSmemFixed + int(sizeof(Bars)) + 1024;
static_assert(kSmemTotal <= 227 * 1024, "shared memory of an SM");

struct ScoreExactArgs {
  const void *Qmax, *Qmin, *Kmax, *Kmin;       // representatives in the workspace
  const float* kabs;                           // [B*Hkv, n2]
  const double* stats;                         // [B,Hq,n1,4]
  const double* S_prev;
  double* S_out;
  DeviceStatus* st;
  int Hq, g, U, n1, n2, seg, blk, segs, n_qchunks, n_combos, fuse, vec;
  int tiles_per_combo, n_tiles;
  double est_scale, ln_alpha, ln_1m_alpha;
};

// d s32, a and b s8, K-major; M = 128, N = 64
constexpr uint32_t kIdesc = (2u << 4) | (1u << 7) | (1u << 10) | (uint32_t(kTileN >> 3) << 17) | (uint32_t(kRows >> 4) << 24);
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p, e;\n.reg .b32 lid;\nelect.sync lid|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
      "@e tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, int* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// The integer a0 + a1 2^8 + ... + a6 2^48, rounded once.  |a_s| <= 2^22.6 (the top digits are at most 64), so the sums of two fit 32
// bits; the low four and the high three become fp64 exactly, through the mantissa of 1.5 x 2^52.
__device__ __forceinline__ double digits_to_f64(int a0, int a1, int a2, int a3, int a4, int a5, int a6) {
  constexpr long long kMagic = 0x4338000000000000ll;
  constexpr double kMagicF = 6755399441055744.0;
  const double lo = __longlong_as_double(mad_wide(a2 + (a3 << 8), 1 << 16, mad_wide(a0 + (a1 << 8), 1, kMagic))) - kMagicF;
  const double hi = __longlong_as_double(mad_wide(a6, 1 << 16, mad_wide(a4 + (a5 << 8), 1, kMagic))) - kMagicF;
  return fma(hi, 4294967296.0, lo);
}

// E with 2^(E-1) <= m < 2^E; kMarked: m is infinite, NaN or so large or small that the scales leave fp32
constexpr int kMarked = 1 << 20;
__device__ __forceinline__ int exponent_of(float m) {
  const int e = int(__float_as_uint(m) >> 23) - 126;
  return m == 0.f ? 30 : (e < -60 || e > 60) ? kMarked : e;
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// 8 elements -> 8 bytes of each digit; true if the row is marked or an element is not a multiple of 2^(E-30)
template <bool kF16>
__device__ __forceinline__ bool to_digits(const uint4& v, int e, uint2 (&out)[kDigits]) {
  const float mul = e == kMarked ? 0.f : __uint_as_float(uint32_t(127 + 30 - e) << 23);
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint32_t dg[8];
  bool bad = e == kMarked;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = unpack2<kF16>(w[i]);
    const float x = f.x * mul, y = f.y * mul;
    const int ix = __float2int_rz(x), iy = __float2int_rz(y);
    bad |= float(ix) != x || float(iy) != y;
    // signed bytes: adding 0x80 to each but the top one carries, the exclusive or takes it off again
    dg[2 * i] = (uint32_t(ix) + 0x00808080u) ^ 0x00808080u;
    dg[2 * i + 1] = (uint32_t(iy) + 0x00808080u) ^ 0x00808080u;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {                // 4 x 4 bytes transposed: digit p of four elements
    const uint32_t* d = dg + 4 * h;
    const uint32_t ab_lo = __byte_perm(d[0], d[1], 0x5140), cd_lo = __byte_perm(d[2], d[3], 0x5140);
    const uint32_t ab_hi = __byte_perm(d[0], d[1], 0x7362), cd_hi = __byte_perm(d[2], d[3], 0x7362);
    const uint32_t p0 = __byte_perm(ab_lo, cd_lo, 0x5410), p1 = __byte_perm(ab_lo, cd_lo, 0x7632);
    const uint32_t p2 = __byte_perm(ab_hi, cd_hi, 0x5410), p3 = __byte_perm(ab_hi, cd_hi, 0x7632);
    if (h == 0) { out[0].x = p0; out[1].x = p1; out[2].x = p2; out[3].x = p3; }
    else { out[0].y = p0; out[1].y = p1; out[2].y = p2; out[3].y = p3; }
  }
  return bad;
}
template <bool kF16>
__device__ __forceinline__ float absmax8(const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  float m = 0.f;
  bool nan = false;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = unpack2<kF16>(w[i]);
    m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
    nan |= f.x != f.x || f.y != f.y;
  }
  return nan ? CUDART_INF_F : m;
}
// 8-byte piece `c` (channels 8 c to 8 c + 7) of row `row` in a 128-byte-swizzled plane of 128-byte rows
__device__ __forceinline__ uint32_t digit_at(int row, int c) { return row * kD + (((c >> 1) ^ (row & 7)) << 4) + (c & 1) * 8; }

// fp64 products of 16 rows with 8 (A and B rows of 128 channels; lane (grp, tig) = (lane / 4, lane % 4) gives A rows grp and grp + 8 and B row grp).
// c: (A row grp, B rows 2 tig, 2 tig + 1), then the same of A row grp + 8.  The order of the channels inside a product is free: a lane takes
// 8 consecutive ones for two MMAs.
template <bool kF16>
__device__ __forceinline__ void exact_16x8(const uint4* a0, const uint4* a1, const uint4* b, int tig, double (&c)[4]) {
  uint4 v0[4], v1[4], vb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { v0[i] = a0[i * 4 + tig]; v1[i] = a1[i * 4 + tig]; vb[i] = b[i * 4 + tig]; }
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 &x = v0[i >> 1], &y = v1[i >> 1], &z = vb[i >> 1];
    const float2 x0 = unpack2<kF16>(i & 1 ? x.z : x.x), x1 = unpack2<kF16>(i & 1 ? x.w : x.y);
    const float2 y0 = unpack2<kF16>(i & 1 ? y.z : y.x), y1 = unpack2<kF16>(i & 1 ? y.w : y.y);
    const float2 z0 = unpack2<kF16>(i & 1 ? z.z : z.x), z1 = unpack2<kF16>(i & 1 ? z.w : z.y);
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7,%8,%9,%10,%11}, {%12,%13,%14,%15}, {%0,%1,%2,%3};"
        : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
        : "d"(double(x0.x)), "d"(double(y0.x)), "d"(double(x0.y)), "d"(double(y0.y)), "d"(double(x1.x)), "d"(double(y1.x)), "d"(double(x1.y)),
          "d"(double(y1.y)), "d"(double(z0.x)), "d"(double(z0.y)), "d"(double(z1.x)), "d"(double(z1.y)));
  }
}

// ln(1 + e^-x), x >= 0, for N independent values: Taylor series around the nearest node, whose coefficients are polynomials in the
// derivative there (gen_softplus_nodes.py; absolute error 1.2e-16).  Written step by step for all N, so that the chains of 19 operations
// run side by side.  The twelve coefficients of a piecewise polynomial, read from shared memory by index, kept that memory busy for
// some 75 cycles per warp and evaluation.
template <int N>
__device__ __forceinline__ void softplus_nodes(const double2* nodes, double (&x)[N]) {
  constexpr double kRound = 211106232532992.0;             // 1.5 x 2^47: sums keep multiples of 1/32
  double s[N], w[N], h[N];
  int at[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    // beyond 40 (infinity and NaN included) as at 40, where f = 4e-18 is below the rounding of what it is added to
    if (uint32_t(__double2hiint(x[i])) >= 0x40440000u) x[i] = 40.0;
    const double y = x[i] + kRound;
    at[i] = __double2loint(y);
    s[i] = nodes[at[i]].y;
    x[i] -= y - kRound;
  }
#pragma unroll
  for (int i = 0; i < N; ++i) w[i] = fma(-s[i], s[i], s[i]);
#pragma unroll
  for (int i = 0; i < N; ++i) h[i] = fma(fma(w[i], 120.0 / 720, -30.0 / 720), w[i], 1.0 / 720);
#pragma unroll
  for (int i = 0; i < N; ++i) h[i] = fma(h[i], x[i], fma(-2.0, s[i], 1.0) * fma(w[i], 12.0 / 120, -1.0 / 120));
#pragma unroll
  for (int i = 0; i < N; ++i) h[i] = fma(h[i], x[i], fma(w[i], -6.0 / 24, 1.0 / 24)) * x[i];
#pragma unroll
  for (int i = 0; i < N; ++i) h[i] = fma(fma(fma(-2.0, s[i], 1.0), -1.0 / 6, h[i]), x[i], 0.5);
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = fma(x[i], fma(w[i] * x[i], h[i], -s[i]), nodes[at[i]].x);
}
// the same by fmax and fmin, which leave a NaN out: for rows and blocks with infinities or NaN
__device__ __forceinline__ double logaddexp_any(const double2* nodes, double a, double b) {
  const double hi = fmax(a, b), lo = fmin(a, b);
  double x[1] = {hi - lo};
  if (!(x[0] >= 0.0)) return hi;
  softplus_nodes(nodes, x);
  return hi + x[0];
}
__device__ __noinline__ double combine_any(const double2* nodes, double L1, double L2, double L3, double L4) {
  const double ln2 = 0.693147180559945309417232121458;
  const double h13 = fmax(L1, L3), h24 = fmax(L2, L4);
  const bool first = h13 >= h24;
  double y = logaddexp_any(nodes, first ? L1 : L2, first ? L3 : L4);
  if (fabs(h13 - h24) < ln2) y = fmax(y, logaddexp_any(nodes, first ? L2 : L1, first ? L4 : L3));
  return y;
}

// max( ln (S1+S3), ln (S2+S4) ) of N scores with finite logits
template <int N>
__device__ __forceinline__ void combine_n(const double2* nodes, const double (&L1)[N], const double (&L2)[N], const double (&L3)[N], const double (&L4)[N],
                                          double (&out)[N]) {
  double hi[2 * N], d[2 * N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    d[i] = L1[i] - L3[i]; d[N + i] = L2[i] - L4[i];
    hi[i] = __double2hiint(d[i]) >= 0 ? L1[i] : L3[i]; hi[N + i] = __double2hiint(d[N + i]) >= 0 ? L2[i] : L4[i];
    d[i] = fabs(d[i]); d[N + i] = fabs(d[N + i]);
  }
  softplus_nodes(nodes, d);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double y13 = hi[i] + d[i], y24 = hi[N + i] + d[N + i];
    out[i] = y13 >= y24 ? y13 : y24;
  }
}
// ln(e^y + e^z) for N scores; fmax and fmin leave a NaN out
template <int N>
__device__ __forceinline__ void fuse_n(const double2* nodes, double (&v)[N], const double (&y)[N], const double (&z)[N]) {
  double d[N];
#pragma unroll
  for (int i = 0; i < N; ++i) { v[i] = fmax(y[i], z[i]); d[i] = v[i] - fmin(y[i], z[i]); }
  softplus_nodes(nodes, d);
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] += d[i];
}

__device__ __forceinline__ void ld4(const double* p, bool vec, int n, double* v) {
  if (vec && n == 4) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = i < n ? p[i] : 0.0;
  }
}
__device__ __forceinline__ void st4(double* p, bool vec, int n, const double* v) {
  if (vec && n == 4) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n) p[i] = v[i];
  }
}

// The row groups and tiles of one CTA: consecutive tiles [lo, hi) of the list (combo, chunk of segments, tile of visible blocks).
struct Walk {
  int at, hi;
  int combo, chunk, tile, n;                   // the current piece: tiles [tile, tile + n) of row group (combo, chunk)
};
__device__ __forceinline__ int visible_of(const ScoreExactArgs& a, int j) { return min(a.n2, ((j + 1) * a.seg + a.blk - 1) / a.blk); }
__device__ __forceinline__ int chunk_tiles(const ScoreExactArgs& a, int chunk) {
  return (visible_of(a, min(a.n1, (chunk + 1) * a.segs) - 1) + kTileBlocks - 1) / kTileBlocks;
}
__device__ __forceinline__ bool next_piece(const ScoreExactArgs& a, Walk& w) {
  if (w.at >= w.hi) return false;
  w.combo = w.at / a.tiles_per_combo;
  int rest = w.at % a.tiles_per_combo;
  int nt;
  for (w.chunk = 0; rest >= (nt = chunk_tiles(a, w.chunk)); ++w.chunk) rest -= nt;
  w.tile = rest;
  w.n = min(nt - rest, w.hi - w.at);
  w.at += w.n;
  return true;
}
// row m of a row group: column m / 8 = (4 segments, head); within it (segment, representative)
struct RowGroup { int kvh, b, h0, j0; };
__device__ __forceinline__ RowGroup row_group(const ScoreExactArgs& a, int combo, int chunk) {
  const int groups = a.g / a.U, Hkv = a.Hq / a.g;
  RowGroup r;
  r.kvh = combo / groups;
  r.b = r.kvh / Hkv;
  r.h0 = (r.kvh % Hkv) * a.g + (combo % groups) * a.U;
  r.j0 = chunk * a.segs;
  return r;
}
__device__ __forceinline__ int row_seg(const ScoreExactArgs& a, const RowGroup& r, int m) {
  return min(a.n1, r.j0 + ((m >> 3) / a.U) * 4 + ((m >> 1) & 3));
}
__device__ __forceinline__ size_t row_unit(const ScoreExactArgs& a, const RowGroup& r, int m) {
  return (size_t(r.b) * a.Hq + r.h0 + (m >> 3) % a.U) * a.n1 + row_seg(a, r, m);
}

// ---------------------------------------------------------------- warps 16-19
template <bool kF16>
__device__ __forceinline__ void convert_role(const ScoreExactArgs& a, Bars* bars, uint8_t* sm, Walk w, int warp, int lane) {
  const int c = lane & 15, half = lane >> 4;   // a warp takes 8 blocks: Kmax rows by the lower half warp, Kmin rows by the upper; 8 channels per lane
  uint32_t t = 0;                              // tiles so far
  while (next_piece(a, w)) {
    const RowGroup r = row_group(a, w.combo, w.chunk);
    const uint4* src = static_cast<const uint4*>(half ? a.Kmin : a.Kmax) + size_t(r.kvh) * a.n2 * (kD / 8) + c;
    const float* abs_src = a.kabs + size_t(r.kvh) * a.n2;
    for (int x = 0; x < w.n; ++x, ++t) {
      const uint32_t stage = t % kStages;
      uint8_t* dst = sm + kSmemK + stage * kDigits * kKPlane;
      Info& info = bars->info[t % kInfo];
      const int blk0 = (w.tile + x) * kTileBlocks + warp * 8;
      uint32_t bad_blocks = 0;
#pragma unroll 1
      for (int i0 = 0; i0 < 8; i0 += 2) {
        uint4 v[2];
        float ka[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const bool in = blk0 + i0 + i < a.n2;
          v[i] = in ? src[size_t(blk0 + i0 + i) * (kD / 8)] : make_uint4(0u, 0u, 0u, 0u);
          ka[i] = in ? abs_src[blk0 + i0 + i] : 0.f;
        }
        if (i0 == 0 && t >= kStages && !mbar_wait(&bars->k_empty[stage], (t / kStages - 1) & 1, &bars->abort_flag, a.st, 71)) return;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int e = exponent_of(ka[i]);
          uint2 dg[kDigits];
          const bool bad = __any_sync(0xffffffffu, to_digits<kF16>(v[i], e, dg));
          const int at = warp * 8 + i0 + i;
#pragma unroll
          for (int p = 0; p < kDigits; ++p) *reinterpret_cast<uint2*>(dst + p * kKPlane + digit_at(half * kTileBlocks + at, c)) = dg[p];
          bad_blocks |= (bad ? 1u : 0u) << (i0 + i);
          if (lane == 0) info.scale[at] = e == kMarked ? 1.0 : pow2(e - 30);
        }
      }
      if (lane == 0) reinterpret_cast<uint8_t*>(&bars->marks[t % kMarks])[warp] = uint8_t(bad_blocks);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the planes through the async proxy
      mbar_arrive(&bars->info_full[t % kInfo]);
      mbar_arrive(&bars->k_full[stage]);
    }
  }
}

// all logit rows are marked: like a tile of marked blocks alone, such tiles are left to redo_marked
__device__ __forceinline__ bool all_marked(const RowInfo& ri) {
  const uint4 v = *reinterpret_cast<const uint4*>(ri.bad);
  return (v.x & v.y & v.z & v.w) == ~0u;
}

// ---------------------------------------------------------------- warp 20
__device__ __forceinline__ void mma_role(const ScoreExactArgs& a, Bars* bars, uint32_t smem, Walk w) {
  const uint32_t tm = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  const uint64_t base = desc_base(16);
  uint32_t t = 0;
  for (uint32_t piece = 0; next_piece(a, w); ++piece) {
    if (!mbar_wait(&bars->q_full, piece & 1, &bars->abort_flag, a.st, 70)) return;
    const bool all_rows = all_marked(bars->rows[piece & 1]);
    for (int x = 0; x < w.n; ++x, ++t) {
      const uint32_t stage = t % kStages;
      if (!mbar_wait(&bars->k_full[stage], (t / kStages) & 1, &bars->abort_flag, a.st, 72)) return;
      if (t > 0 && !mbar_wait(&bars->acc_empty, (t - 1) & 1, &bars->abort_flag, a.st, 73)) return;
      tc_fence_after();
      const uint32_t k_smem = smem + kSmemK + stage * kDigits * kKPlane;
      if (!all_rows && bars->marks[t % kMarks] != ~0u) {
#pragma unroll
        for (int s = 0; s < kAccs; ++s)
#pragma unroll
          for (int i = s > 3 ? s - 3 : 0; i <= (s < 3 ? s : 3); ++i)
#pragma unroll
            for (int kk = 0; kk < kD / 32; ++kk)
              umma_i8(tm + s * kTileN, desc_at(base, smem + i * kQPlane + kk * 32), desc_at(base, k_smem + (s - i) * kKPlane + kk * 32),
                      i > (s > 3 ? s - 3 : 0) || kk > 0);
      }
      umma_commit(&bars->acc_full);
      umma_commit(&bars->k_empty[stage]);
    }
  }
}

// ---------------------------------------------------------------- warps 0-15
// The scores of a row group's marked blocks and of its marked rows once more, from fp64 products; t: the CTA's tiles up to the end of the group.  An MMA tile
// is 8 blocks (Kmax, Kmin) with 4 pairs of rows (Qmax, Qmin) of a (head, segment): each lane then holds the four logits of a score.  Marked
// blocks are gathered over the whole group, so that few of them cost little: 8 with 64 pairs take 4100 cycles of the fp64 pipes.  Returns how
// often the epilogue warps have met here by then.
constexpr uint32_t kGaveUp = ~0u;
template <bool kF16>
__device__ __forceinline__ uint32_t redo_marked(const ScoreExactArgs& a, Bars* bars, int combo, int chunk, int tile, int n_tiles, uint32_t piece, uint32_t t,
                                             uint32_t redone) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane >> 2, tig = lane & 3;
  const RowInfo& ri = bars->rows[piece & 1];
  const uint32_t t0 = t - n_tiles;
  int n_blocks = 0;                            // marked blocks; bits of the lanes' words first
  for (int i = lane; i < n_tiles; i += 32) n_blocks += __popc(bars->marks[(t0 + i) % kMarks]);
  n_blocks = __reduce_add_sync(0xffffffffu, n_blocks);
  const uint32_t* row_words = reinterpret_cast<const uint32_t*>(ri.bad);
  auto pair_marked = [&](int p) { return (row_words[p >> 4] >> (2 * (p & 15)) & 3u) != 0; };
  const uint32_t pairs_lo = __ballot_sync(0xffffffffu, pair_marked(lane)), pairs_hi = __ballot_sync(0xffffffffu, pair_marked(32 + lane));
  int n_pairs = __popc(pairs_lo) + __popc(pairs_hi);
  if (n_blocks + n_pairs == 0) return redone;
  const int first = tile * kTileBlocks, in_group = min(n_tiles * kTileBlocks, a.n2 - first);
  // all pairs with the marked blocks, then the marked pairs with all blocks; or, where that is no more, all with all
  const int all_units = (kRows / 8) * ((in_group + 7) / 8);
  int block_units = (kRows / 8) * ((n_blocks + 7) / 8);
  const bool whole = block_units + (n_pairs + 3) / 4 * ((in_group + 7) / 8) >= all_units;
  if (whole) { block_units = 0; n_pairs = kRows / 2; }
  if (warp == 0) {                             // the lists; nobody reads those of the group before any more: all have passed the wait for q_full
    int at = 0;
    for (int i0 = 0; i0 < n_tiles && !whole; i0 += 32) {
      uint32_t word = i0 + lane < n_tiles ? bars->marks[(t0 + i0 + lane) % kMarks] : 0u;
      int incl = __popc(word);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
      }
      int pos = at + incl - __popc(word);
      for (; word; word &= word - 1) bars->redo_blocks[pos++] = uint16_t((i0 + lane) * kTileBlocks + __ffs(word) - 1);
      at += __shfl_sync(0xffffffffu, incl, 31);
    }
    const uint32_t below = (1u << lane) - 1u;
    if (whole || (pairs_lo >> lane & 1u)) bars->redo_pairs[whole ? lane : __popc(pairs_lo & below)] = uint8_t(lane);
    if (whole || (pairs_hi >> lane & 1u)) bars->redo_pairs[whole ? 32 + lane : __popc(pairs_lo) + __popc(pairs_hi & below)] = uint8_t(32 + lane);
  }
  // what is stored below overwrites what other threads have stored for these scores
  mbar_arrive(&bars->redo);
  if (!mbar_wait(&bars->redo, redone++ & 1, &bars->abort_flag, a.st, 77)) return kGaveUp;

  const RowGroup r = row_group(a, combo, chunk);
  const int pair_units = (n_pairs + 3) / 4, units = block_units + pair_units * ((in_group + 7) / 8);
#pragma unroll 1
  for (int u = warp; u < units; u += kEpilogueWarps) {
    const bool by_block = u < block_units;
    const int n_groups = by_block ? kRows / 8 : pair_units, v = by_block ? u : u - block_units;
    const int pg = v % n_groups * 4, bg = v / n_groups * 8 + grp;           // the unit's first pair; the lane's block
    auto pair_at = [&](int i) { return by_block ? i : int(bars->redo_pairs[min(i, n_pairs - 1)]); };
    const int block = first + (by_block ? int(bars->redo_blocks[min(bg, n_blocks - 1)]) : min(bg, in_group - 1));
    const int mq = 2 * pair_at(pg + (grp >> 1)) + (grp & 1), ms = 2 * pair_at(pg + tig);    // the lane's B row; Qmax row of its score
    const int j = row_seg(a, r, ms);
    const bool here = j < a.n1 && (by_block ? bg < n_blocks : bg < in_group && pg + tig < n_pairs), seen = here && block < visible_of(a, j);
    const size_t key = (size_t(r.kvh) * a.n2 + block) * (kD / 8), at = (here ? row_unit(a, r, ms) : 0) * a.n2 + block;
    const double sp = a.fuse && seen ? a.S_prev[at] : 0.0;
    double c[4];
    exact_16x8<kF16>(static_cast<const uint4*>(a.Kmax) + key, static_cast<const uint4*>(a.Kmin) + key,
                     static_cast<const uint4*>((mq & 1) ? a.Qmin : a.Qmax) + (row_seg(a, r, mq) < a.n1 ? row_unit(a, r, mq) : 0) * (kD / 8), tig, c);
    const double L1[1] = {fma(c[0], a.est_scale, -ri.lse[ms][0])}, L2[1] = {fma(c[2], a.est_scale, -ri.lse[ms][1])};
    const double L3[1] = {fma(c[1], a.est_scale, -ri.lse[ms + 1][0])}, L4[1] = {fma(c[3], a.est_scale, -ri.lse[ms + 1][1])};
    const bool finite = fabs(L1[0]) < CUDART_INF && fabs(L2[0]) < CUDART_INF && fabs(L3[0]) < CUDART_INF && fabs(L4[0]) < CUDART_INF;
    double s[1];
    if (__all_sync(0xffffffffu, finite)) combine_n(bars->nodes, L1, L2, L3, L4, s);
    else s[0] = combine_any(bars->nodes, L1[0], L2[0], L3[0], L4[0]);
    s[0] -= 0.693147180559945309417232121458;
    if (a.fuse) {
      const double y[1] = {a.ln_alpha + s[0]}, z[1] = {a.ln_1m_alpha + sp};
      fuse_n(bars->nodes, s, y, z);
    }
    if (here) a.S_out[at] = seen ? s[0] : -CUDART_INF;
  }
  return redone;
}

template <bool kF16>
__device__ __forceinline__ void epilogue_role(const ScoreExactArgs& a, Bars* bars, uint8_t* sm, Walk w, int warp, int lane) {
  const int m = (warp & 3) * 32 + lane, hc = warp >> 2;     // logit row; quarter of the tile's blocks
  const uint32_t tm = bars->tmem_base + (uint32_t((warp & 3) * 32) << 16) + hc * 8;
  const bool odd = lane & 1;                                // Qmin rows; the lane takes the upper 4 of its 8 blocks
  const double ln2 = 0.693147180559945309417232121458;
  uint32_t t = 0, redone = 0;
  for (uint32_t piece = 0; next_piece(a, w); ++piece) {
    const RowGroup r = row_group(a, w.combo, w.chunk);
    RowInfo& ri = bars->rows[piece & 1];
    {
      // The bytes of the row group's query rows, 8 rows per warp, two at a time.  The MMAs on the row group before have all been
      // completed: this warp has seen the last of them.
      const int c = lane & 15, m0 = (warp & 3) * 32 + hc * 8 + (lane >> 4);
      uint4 q[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int mq = m0 + 2 * i;
        q[i] = make_uint4(0u, 0u, 0u, 0u);
        if (row_seg(a, r, mq) < a.n1) q[i] = static_cast<const uint4*>((mq & 1) ? a.Qmin : a.Qmax)[row_unit(a, r, mq) * (kD / 8) + c];
      }
      uint32_t bad_rows = 0;
      bool not_finite = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int mq = m0 + 2 * i;
        float mx = absmax8<kF16>(q[i]);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int e = exponent_of(mx);
        uint2 dg[kDigits];
        const unsigned bad = __ballot_sync(0xffffffffu, to_digits<kF16>(q[i], e, dg));
#pragma unroll
        for (int p = 0; p < kDigits; ++p) *reinterpret_cast<uint2*>(sm + p * kQPlane + digit_at(mq, c)) = dg[p];
        const uint32_t both = ((bad & 0xffffu) != 0 ? 1u : 0u) | ((bad >> 16) != 0 ? 2u : 0u);
        bad_rows |= both << (2 * i);
        if (c < 2) {
          const double l = row_seg(a, r, mq) < a.n1 ? a.stats[row_unit(a, r, mq) * 4 + 2 * (mq & 1) + c] : 0.0;
          ri.lse[mq][c] = l;
          not_finite |= !(fabs(l) < CUDART_INF);
        }
        if (c == 0) ri.scale[mq] = e == kMarked ? 1.0 : pow2(e - 30);
      }
      not_finite = __any_sync(0xffffffffu, not_finite);
      if (lane == 0) { ri.bad[(warp & 3) * 4 + hc] = uint8_t(bad_rows); ri.special[(warp & 3) * 4 + hc] = not_finite; }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the planes through the async proxy
      mbar_arrive(&bars->q_full);
    }
    const int j = row_seg(a, r, m);
    const bool valid = j < a.n1;
    const size_t unit = row_unit(a, r, m);
    const int vis = valid ? visible_of(a, j) : 0;
    const int warp_vis = __reduce_max_sync(0xffffffffu, vis);
    if (!mbar_wait(&bars->q_full, piece & 1, &bars->abort_flag, a.st, 76)) return;
    const bool all_rows = all_marked(ri);
    const bool special = *reinterpret_cast<const uint32_t*>(&ri.special[(warp & 3) * 4]) != 0;
    for (int x = 0; x < w.n; ++x, ++t) {
      const int b_tile = (w.tile + x) * kTileBlocks + hc * 8, b0 = b_tile + (odd ? 4 : 0);
      const int n_in = valid ? min(4, a.n2 - b0) : 0;       // blocks of this lane that exist
      const size_t out = unit * a.n2 + b0;
      double sp[4];
      const bool any = b_tile < warp_vis;                   // some row of the warp sees some of its 8 blocks
      if (a.fuse && any) ld4(a.S_prev + out, a.vec, n_in, sp);
      if (!mbar_wait(&bars->info_full[t % kInfo], (t / kInfo) & 1, &bars->abort_flag, a.st, 74)) return;
      if (!mbar_wait(&bars->acc_full, t & 1, &bars->abort_flag, a.st, 75)) return;
      tc_fence_after();
      if (all_rows || bars->marks[t % kMarks] == ~0u) {     // every score of the tile follows from redo_marked
        tc_fence_before();
        mbar_arrive(&bars->acc_empty);
        continue;
      }
      if (!any) {
        tc_fence_before();
        mbar_arrive(&bars->acc_empty);
        const double v[4] = {-CUDART_INF, -CUDART_INF, -CUDART_INF, -CUDART_INF};
        st4(a.S_out + out, a.vec, n_in, v);
        continue;
      }
      const Info& info = bars->info[t % kInfo];
      double vx[8], vn[8];                                  // integer dot products with the Kmax / Kmin rows of the 8 blocks
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        const uint32_t col = tm + (part >> 1) * kTileBlocks + (part & 1) * 4;
        int acc[kAccs][4];
#pragma unroll
        for (int s = 0; s < kAccs; ++s) tmem_ld4(col + s * kTileN, acc[s]);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double d = digits_to_f64(acc[0][i], acc[1][i], acc[2][i], acc[3][i], acc[4][i], acc[5][i], acc[6][i]);
          if (part < 2) vx[(part & 1) * 4 + i] = d; else vn[(part & 1) * 4 + i] = d;
        }
      }
      tc_fence_before();
      mbar_arrive(&bars->acc_empty);
      // The Qmax lane gives its upper blocks for the Qmin lane's lower ones: each then has all four logits of 4 blocks, less
      // their log-sum-exps.  Which of a pair is l1 (l2) and which l3 (l4) makes no difference.
      const double f_own = ri.scale[m] * a.est_scale, f_other = ri.scale[m ^ 1] * a.est_scale;
      const double2 lse_own = *reinterpret_cast<const double2*>(ri.lse[m]), lse_other = *reinterpret_cast<const double2*>(ri.lse[m ^ 1]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double ox = __shfl_xor_sync(0xffffffffu, odd ? vx[i] : vx[4 + i], 1), on = __shfl_xor_sync(0xffffffffu, odd ? vn[i] : vn[4 + i], 1);
        const double mx = odd ? vx[4 + i] : vx[i], mn = odd ? vn[4 + i] : vn[i];
        const double bs = info.scale[hc * 8 + (odd ? 4 : 0) + i];
        const double fm = f_own * bs, fo = f_other * bs;
        vx[i] = fma(mx, fm, -lse_own.x); vn[i] = fma(mn, fm, -lse_own.y);
        vx[4 + i] = fma(ox, fo, -lse_other.x); vn[4 + i] = fma(on, fo, -lse_other.y);
      }
      // max( ln (S1+S3)/2, ln (S2+S4)/2 ), fusion with S'
      double v[4];
      if (special) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = combine_any(bars->nodes, vx[i], vn[i], vx[4 + i], vn[4 + i]) - ln2;
      } else {
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          const double L1[2] = {vx[q], vx[q + 1]}, L2[2] = {vn[q], vn[q + 1]}, L3[2] = {vx[4 + q], vx[5 + q]}, L4[2] = {vn[4 + q], vn[5 + q]};
          double y[2];
          combine_n(bars->nodes, L1, L2, L3, L4, y);
          v[q] = y[0] - ln2; v[q + 1] = y[1] - ln2;
        }
      }
      if (a.fuse) {
        double y[4], z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { y[i] = a.ln_alpha + v[i]; z[i] = a.ln_1m_alpha + sp[i]; }
        fuse_n(bars->nodes, v, y, z);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = b0 + i < vis ? v[i] : -CUDART_INF;     // blocks at or after the end of the segment (line 13)
      st4(a.S_out + out, a.vec, n_in, v);
    }
    redone = redo_marked<kF16>(a, bars, w.combo, w.chunk, w.tile, w.n, piece, t, redone);
    if (redone == kGaveUp) return;
  }
}

// ---------------------------------------------------------------- warps 21-23: blocks after the tiles of a row group
__device__ __forceinline__ void mask_role(const ScoreExactArgs& a, int warp, int lane) {
  const size_t rows = size_t(a.n_combos) * a.U * a.n1;      // = batch x heads x segments
  for (size_t u = size_t(blockIdx.x) * 3 + warp; u < rows; u += size_t(gridDim.x) * 3) {
    const int lo = chunk_tiles(a, int(u % a.n1) / a.segs) * kTileBlocks;
    double* row = a.S_out + u * a.n2;
    if (a.vec) {
      for (int b = lo + lane * 4; b < a.n2; b += 128)
        asm volatile("st.global.v4.f64 [%0], {%1, %1, %1, %1};" ::"l"(row + b), "d"(-CUDART_INF) : "memory");
    } else {
      for (int b = lo + lane; b < a.n2; b += 32) row[b] = -CUDART_INF;
    }
  }
}

template <bool kF16>
__global__ void __launch_bounds__(kThreads, 1) score_visible_kernel(const __grid_constant__ ScoreExactArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t smem_base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (smem_base - raw);
  Bars* bars = reinterpret_cast<Bars*>(sm + kSmemFixed);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&bars->k_full[i], 128); mbar_init(&bars->k_empty[i], 1); }
    for (int i = 0; i < kInfo; ++i) mbar_init(&bars->info_full[i], 128);
    mbar_init(&bars->q_full, kEpilogueWarps * 32);
    mbar_init(&bars->acc_full, 1);
    mbar_init(&bars->acc_empty, kEpilogueWarps * 32);
    mbar_init(&bars->redo, kEpilogueWarps * 32);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) { tmem_alloc(&bars->tmem_base, 512); tmem_relinquish(); }
  for (int e = tid; e < kNodes; e += kThreads) bars->nodes[e] = kSoftplusNodes[e];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  pdl_wait();                                  // the loads behind it are plain ones, which stay behind it

  Walk w;
  w.at = int((long long)a.n_tiles * blockIdx.x / gridDim.x);
  w.hi = int((long long)a.n_tiles * (blockIdx.x + 1) / gridDim.x);
  static_assert(kRegPoolNeeded <= kThreads * 80, "setmaxnreg budget exceeds the launch allocation");
  if (warp < kEpilogueWarps) {
    reg_inc<kEpilogueRegs>();
    epilogue_role<kF16>(a, bars, sm, w, warp, lane);
  } else {
    reg_dec<kOtherRegs>();
    if (warp < kMmaWarp) convert_role<kF16>(a, bars, sm, w, warp - kEpilogueWarps, lane);
    else if (warp == kMmaWarp) mma_role(a, bars, smem_base, w);
    else mask_role(a, warp - kMmaWarp - 1, lane);
  }
  if (bars->abort_flag) {
    for (int i = 0; i < 200; ++i) __nanosleep(1000);        // let MMAs in flight land before the CTA's resources go
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(bars->tmem_base, 512);
}

template <bool kF16>
int launch_visible(const Dims& m, char* ws, const double* S_prev, double* S_out, double est_scale, double alpha, int fuse, cudaStream_t st) {
  const WsLayout w = ws_layout(m);
  ScoreExactArgs a;
  a.Qmax = ws + w.qmax; a.Qmin = ws + w.qmin; a.Kmax = ws + w.kmax; a.Kmin = ws + w.kmin;
  a.kabs = reinterpret_cast<const float*>(ws + w.kabs);
  a.stats = reinterpret_cast<const double*>(ws + w.stats);
  a.S_prev = S_prev; a.S_out = S_out;
  a.st = reinterpret_cast<DeviceStatus*>(ws);
  a.Hq = m.Hq; a.g = m.g; a.U = score_heads(m);
  a.n1 = m.n1; a.n2 = m.n2; a.seg = m.seg; a.blk = m.blk;
  a.segs = 64 / a.U;
  a.n_qchunks = (m.n1 + a.segs - 1) / a.segs;
  a.n_combos = m.B * m.Hkv * (m.g / a.U);
  a.fuse = fuse;
  // whole 32-byte sectors where every row of the map starts on one
  a.vec = m.n2 % 4 == 0 && (reinterpret_cast<uintptr_t>(S_out) & 31u) == 0 && (!fuse || (reinterpret_cast<uintptr_t>(S_prev) & 31u) == 0);
  long long per_combo = 0;
  for (int c = 0; c < a.n_qchunks; ++c) {
    const int j = (c + 1) * a.segs < m.n1 ? (c + 1) * a.segs - 1 : m.n1 - 1;
    const long long end = ((long long)(j + 1) * m.seg + m.blk - 1) / m.blk;
    per_combo += ((end < m.n2 ? end : m.n2) + kTileBlocks - 1) / kTileBlocks;
  }
  if (per_combo * a.n_combos > 0x7fffffffLL) return CP_ERR_UNSUPPORTED;
  a.tiles_per_combo = int(per_combo);
  a.n_tiles = int(per_combo * a.n_combos);
  a.est_scale = est_scale; a.ln_alpha = log(alpha); a.ln_1m_alpha = log1p(-alpha);
  auto kern = score_visible_kernel<kF16>;
  // setmaxnreg.inc blocks forever when the registers that the kernel was compiled to are fewer than what the roles ask for: refuse
  // to launch such a build instead
  static int regs_ok = 0;
  if (regs_ok == 0) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return CP_ERR_CUDA;
    regs_ok = fa.numRegs * kThreads >= kRegPoolNeeded ? 1 : -1;
  }
  if (regs_ok < 0) return CP_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal) != cudaSuccess) return CP_ERR_CUDA;
  const unsigned grid = unsigned(a.n_tiles < 148 ? a.n_tiles : 148);   // one CTA per SM
  return launch_pdl(kern, dim3(grid), kThreads, kSmemTotal, st, a);
}

}  // namespace

// Whether the two-kernel path is the faster one, by estimates of both (us).  The general kernel's work is its (CTA, key block) pairs per SM, which single heads
// use no better than groups of four.  The two kernels start with some 36 us; the log-sum-exps take time for every wave of CTAs, by the key blocks that
// each of them streams and by the share of its 128 rows that is in use; the visible blocks by their tiles per SM.  From 2.2 M scores on
// two kernels are taken whatever the shape.  Fitted to 538 shapes (0.2 to 3.2 M scores, groups of 1 to 8 heads, segments of 128 to 1024, blocks of
// 32 to 128, fused and not) with clustered keys as in attention, and with keys of which ten times as many come near a row's maximum: 0.8 and 2.0 %
// slower on average than the better path of each.  A line at 1.5 M scores, those of groups of 2 heads counted twice and of single heads and
// odd groups four times: 2.6 and 6.8 %, up to 1.4 and 1.9 times.
// General kernel / two kernels, us, fused, clustered keys: 32 / 8 heads, segment 512, block 32, 15995 tokens 39.5 / 66.8, 27707 tokens 105.0 / 106.4, 33531
// tokens 154.5 / 124.4; segment 1024, block 128, 84603 tokens 131.2 / 142.5; 24 / 8 heads, segment 512, block 64, 28603 tokens 112.4 / 96.5.
constexpr long long kFastMinScores = 2200000;
bool score_is_split(const cp_params& p, const Dims& m) {
  if ((p.dtype != CP_BF16 && p.dtype != CP_F16) || m.d != 128) return false;
  if ((p.flags & CP_FLAG_FORCE_SPLIT_SCORE) || (long long)m.B * m.Hq * m.n1 * m.n2 >= kFastMinScores) return true;
  const int U = score_heads(m), segs = lse_segments(m);
  const long long groups = (long long)m.B * m.Hkv * (m.g / U);
  const double per_sm = double(groups) * m.n1 * m.n2 / 148, waves = double((groups * ((m.n1 + segs - 1) / segs) + 147) / 148);
  const double general = 16 + (0.019 + 0.0045 * U) * per_sm;
  const double split = 36 + waves * (10 + m.n2 * (0.025 + 0.14 * segs * U / 64)) + 7.5 / 4096 * U * per_sm;
  return general > split;
}

// K2 dispatcher.  16-bit inputs with head_dim 128 take the two-kernel path (log-sum-exps, then exact logits of
// the visible blocks); everything else the general kernel.
int launch_score(const cp_params& p, const Dims& m, char* ws, const double* S_prev, double* S_out, cudaStream_t st) {
  // The two-kernel path pays for an extra launch and for the serial sweeps of the log-sum-exp kernel; it wins once the
  // score map is large, so small maps keep the general kernel.
  if (!score_is_split(p, m)) return launch_score_generic(p, m, ws, S_prev, S_out, nullptr, st);
  const int rc = launch_lse(p, m, ws, st);
  if (rc != CP_OK) return rc;
  const int fuse = (S_prev != nullptr && p.alpha != 1.0f) ? 1 : 0;
  const double es = double(p.est_scale), al = double(p.alpha);
  return p.dtype == CP_F16 ? launch_visible<true>(m, ws, S_prev, S_out, es, al, fuse, st)
                           : launch_visible<false>(m, ws, S_prev, S_out, es, al, fuse, st);
}

}  // namespace cp
