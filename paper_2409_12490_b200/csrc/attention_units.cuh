// Work units of the tensor-core attention kernels (attention_sm100.cu, attention_pair_sm100.cu): their order, the tiles they stream,
// and the check of their block lists.
#pragma once
#include "sm100_ptx.cuh"

namespace cp {

// One work unit, decoded (the scheduler warp decodes it once and publishes it to the other warps:
// the decoding is a chain of integer divisions that would otherwise sit at the start of every unit).
struct Unit {
  int b, h, kvh;
  int seq;          // sequence of a packed batch (0 for a single problem)
  int n;            // its length
  int q_tok;        // first query row of tile A
  int n_past;       // listed blocks strictly before the segment
  int n_past_tiles; // gathered tiles
  int last_cols;    // valid key columns of the last gathered tile
  int c_tok, n_cont;// contiguous unmasked tiles: first token, count
  int d_tok;        // first token of diagonal tile d0 (d1 follows)
  int T;            // K/V tiles the unit streams
  int nA, nB;       // tiles query tile A / B consumes (nB = 0: the unit has no tile B)
  const int32_t* list;
  int seg_j;
  int rj;           // diagonal blocks of the segment (r, fewer in a short last segment)
  int cnt;
  int generic;      // the list is not "past blocks, then exactly the diagonal blocks": every listed block is gathered and
                    // every tile is masked element by element (a key counts iff its token is not after the query's)
  int rowsB;        // the unit has a second 128-row query tile
};

// One sequence: where its tokens, lists and rows of lse start in the arrays of the launch.
struct Seq {
  int n, n1, n2;
  int seg0;                     // segments of the sequences before it
  int64_t tok0, idx0, cnt0, lse0;
};
constexpr int kMaxSeqs = 16;
constexpr int kMaxOrder = 1024;

template <int NS> struct Args {
  const int32_t* idx;
  const int32_t* cnt;
  uint16_t* O;                  // bf16 or fp16 elements
  float* lse;
  DeviceStatus* st;
  int B, Hq, Hkv, g, seg, blk, k, r;
  int pp;                       // units (pairs of query tiles) per segment, counted over the rows that a segment can have
  int64_t osb, osh, ost;
  const uint16_t *Q, *K, *V;    // only for rows that are evaluated one by one (exact_row)
  int64_t qs[3], ks[3], vs[3];
  float sm_scale;
  int dense;
  int n_units;
  int n_seqs, n_segs;           // sequences, segments of all sequences
  int long_first;               // order of the units: see decode_unit
  Seq seq[NS];
  uint16_t order[kMaxOrder];    // long_first, not dense: (segment * pairs per segment + pair), longest units first
  int o_vec32;                  // O rows are 32-byte aligned: the epilogue may use 32-byte stores
  int emul;                     // long units: part of the exponentials on the FMA pipes (see launch_attention_sm100)
  int withhold_v;               // test hook: the producer never issues V tiles, so a bounded wait must expire
};
// tensor maps of each sequence; the launch's tensors have up to 4 dimensions, kQ .. kVt name their boxes
enum { kQ = 0, kKb = 1, kVb = 2, kKt = 3, kVt = 4, kMaps = 5 };   // query tile, K / V block, K / V tile
template <int NS> struct Maps { CUtensorMap m[NS][kMaps]; };
template <int NS> struct OMaps { CUtensorMap m[NS]; };            // 32 rows of O

namespace {

constexpr int kTile = 128;
constexpr int kHalfBytes = kTile * 64 * 2;   // [128 rows x 64 cols] of 16-bit elements, 128-byte swizzled
constexpr float kRescaleThreshold = 8.0f;    // in log2 units
#ifndef CP_EMUL_EVERY
#define CP_EMUL_EVERY 8
#endif
constexpr int kEmulEvery = CP_EMUL_EVERY;    // launches of long units: every n-th pair of exponentials on the FMA pipes (0: none)

// ---------------------------------------------------------------- unit geometry

// Units of a segment or of a long sequence share K/V tiles with the other query heads of their KV head, so units are
// ordered KV-head-major (within a KV head from the sequence's end, longest first for the dense kernel): the CTAs that are
// resident together then read the same tiles through L2.  When all K and V (nearly) fit L2 together that does not matter
// and the order is longest units first over all heads and sequences (long_first; the host sorts the (segment, pair)s by
// the tiles they stream), which leaves the short ones to even out the ends of the CTAs.  Both orders, us, 32 query / 8 KV heads:
// dense, KV-head-major / longest first: 34 MB of K and V 592 / 502, 101 MB 4479 / 4367, 168 MB 12125 / 12106, 201 MB 17344 / 17439,
// 268 MB 30381 / 31149; segment 512, budget 1024: 67 MB 267 / 247, 134 MB 539 / 504, 268 MB 1069 / 1007, 537 MB 2113 / 2039; segment
// 1024, budget 4096: 134 MB 1783 / 1749, 268 MB 3647 / 3586, 537 MB 7335 / 7285.  The line (160 MB) is the dense kernel's.
// `cnt` is the unit's list length when the caller already has it, kLoadCnt to read it from global memory.
constexpr int kLoadCnt = -2, kBadList = -1, kEmptyUnit = -3, kZeroUnit = -4;   // kEmptyUnit: no query row of the unit lies inside the sequence;
                                                                                // kZeroUnit: an empty list -- the unit's rows are zeros
template <int NS>
__device__ __forceinline__ Unit decode_unit(const Args<NS>& a, int x, int cnt) {
  Unit u;
  u.list = nullptr;
  u.cnt = 0;
  u.seq = 0;
  u.n = a.seq[0].n;
  if (a.dense) {
    const int ntiles = (u.n + kTile - 1) / kTile;
    const int np = (ntiles + 1) / 2;
    int pair;
    if (a.long_first) {
      const int heads = a.B * a.Hq, bh = x % heads;
      pair = np - 1 - x / heads;
      u.b = bh / a.Hq; u.h = bh % a.Hq; u.kvh = u.h / a.g;
    } else {
      const int per_kvh = a.g * np;
      const int bkv = x / per_kvh;
      const int rest = x - bkv * per_kvh;
      pair = np - 1 - rest / a.g;
      u.b = bkv / a.Hkv; u.kvh = bkv % a.Hkv; u.h = u.kvh * a.g + rest % a.g;
    }
    u.q_tok = pair * 256;
    u.n_past = 0; u.n_past_tiles = 0; u.last_cols = kTile;
    u.c_tok = 0; u.n_cont = 2 * pair; u.d_tok = pair * 256;
    u.seg_j = 0; u.rj = 0;
    u.nB = (2 * pair + 1 < ntiles) ? 1 : 0;
  } else {
    const int q_tiles = a.seg / kTile;
    const int pp = a.pp;
    int j, p;
    if (a.long_first) {
      const int heads = a.B * a.Hq, bh = x % heads;
      const int y = a.order[x / heads];
      j = y / pp;
      p = y % pp;
      if constexpr (NS > 1) {
        while (u.seq + 1 < a.n_seqs && j >= a.seq[u.seq + 1].seg0) ++u.seq;
        j -= a.seq[u.seq].seg0;
        u.n = a.seq[u.seq].n;
      }
      u.b = bh / a.Hq; u.h = bh % a.Hq; u.kvh = u.h / a.g;
    } else {
      const int gi_p = a.g * pp;
      const int per_kvh = a.n_segs * gi_p;
      const int bkv = x / per_kvh;
      const int rest = x - bkv * per_kvh;
      j = a.n_segs - 1 - rest / gi_p;
      p = rest % pp;
      u.b = bkv / a.Hkv; u.kvh = bkv % a.Hkv; u.h = u.kvh * a.g + (rest % gi_p) / pp;
    }
    const Seq& sq = a.seq[u.seq];
    u.seg_j = j;
    u.q_tok = j * a.seg + p * 256;
    const long long unit = ((long long)u.b * a.Hq + u.h) * sq.n1 + j;
    u.list = a.idx + sq.idx0 + unit * a.k;
    u.cnt = cnt == kLoadCnt ? a.cnt[sq.cnt0 + unit] : cnt;
    u.rj = min(sq.n2, (j + 1) * a.r) - j * a.r;
    u.n_past = min(max(u.cnt - u.rj, 0), a.k);
    u.n_past_tiles = (u.n_past * a.blk + kTile - 1) / kTile;
    u.last_cols = u.n_past * a.blk - (u.n_past_tiles - 1) * kTile;
    u.c_tok = j * a.seg; u.n_cont = 2 * p; u.d_tok = u.q_tok;
    u.nB = (2 * p + 1 < q_tiles && u.q_tok + kTile < u.n) ? 1 : 0;   // tile B exists and starts inside the sequence
  }
  u.generic = 0;
  u.rowsB = u.nB ? 1 : 0;
  u.nA = u.n_past_tiles + u.n_cont + 1;       // up to and including its own diagonal tile
  u.nB = u.nB ? u.nA + 1 : 0;                 // one more diagonal tile; 0 when the segment has an odd tile count
  u.T = u.nB ? u.nB : u.nA;
  return u;
}

// The list contract, checked by the scheduler warp before it publishes a unit: at most k entries, ascending, unique,
// each a block the segment can see (0 <= b < (j+1)*r).  Returns 0 when the list has the form the selection emits
// (past blocks, then exactly the diagonal blocks of the segment: the fast tile sequence applies), 1 for any other
// valid list (generic tile sequence), -1 for a list that breaks the contract.
template <int NS>
__device__ __forceinline__ int classify_unit(const Args<NS>& a, const Unit& u, int lane) {
  if (a.dense) return 0;
  const int vis = min(a.seq[u.seq].n2, (u.seg_j + 1) * a.r);
  bool gen_ok = (u.cnt >= 0) && (u.cnt <= a.k);
  bool std_ok = gen_ok && (u.cnt >= u.rj);
  if (gen_ok) {
    for (int i = lane; i < u.cnt; i += 32) {
      const int v = u.list[i];
      const bool asc = v >= 0 && v < vis && (i == 0 || u.list[i - 1] < v);
      gen_ok = gen_ok && asc;
      if (i >= u.n_past) std_ok = std_ok && (v == u.seg_j * a.r + (i - u.n_past));
      else std_ok = std_ok && asc && v < u.seg_j * a.r;
    }
  }
  gen_ok = __all_sync(0xffffffffu, gen_ok);
  std_ok = __all_sync(0xffffffffu, std_ok);
  return !gen_ok ? -1 : (std_ok ? 0 : 1);
}

template <int NS, typename Bars>
__device__ __forceinline__ bool stop_requested(const Args<NS>& a, Bars* bars) {
  return bars->abort_flag || (a.st != nullptr && *reinterpret_cast<volatile int32_t*>(&a.st->code) == CP_ERR_TIMEOUT);
}

// The unit with index x, decoded and its list checked, by a whole warp; its cnt is the list's length or one of the codes above.
// A list that breaks its contract is published with length kBadList and skipped by everyone.  (attention_sm100.cu has this in its
// scheduler, as its masks in its softmax role: out of there, long loops over long units were 1 to 2 % slower.)
template <int NS>
__device__ __forceinline__ Unit prepare_unit(const Args<NS>& a, int x, int lane) {
  Unit u = decode_unit(a, x, kLoadCnt);
  int cnt = u.cnt;
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
  u.cnt = cnt;
  return u;
}

// an empty list: no key is visible to any row of the unit -- zeros, and lse = ln 0
template <int D, int NS>
__device__ __forceinline__ void write_zero_row(const Args<NS>& a, const Unit& u, int which, int t) {
  if ((which == 0 || u.rowsB) && t < u.n) {
    uint4* dst = reinterpret_cast<uint4*>(a.O + u.b * a.osb + u.h * a.osh + (a.seq[u.seq].tok0 + t) * a.ost);
#pragma unroll
    for (int i = 0; i < D * 2 / 16; ++i) dst[i] = make_uint4(0u, 0u, 0u, 0u);
    if (a.lse != nullptr) a.lse[a.seq[u.seq].lse0 + ((long long)u.b * a.Hq + u.h) * u.n + t] = -CUDART_INF;
  }
}

}  // namespace

// attention_pair_sm100.cu, for launches whose maps have its boxes
template <int NS> int launch_attention_pair(const Maps<NS>& maps, const OMaps<NS>& o_maps, const Args<NS>& a, bool f16, cudaStream_t s);

}  // namespace cp
