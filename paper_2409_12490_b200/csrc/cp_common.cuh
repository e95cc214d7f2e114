// Shared host/device declarations of the CUDA path (not used by the CPU oracle).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "critiprefill.h"

namespace cp {

constexpr int kStatusBytes = 256;   // head of the workspace: status word + diagnostics
constexpr int kMaxBlocksN2 = 8192;  // estimate: fp64 logits in the shared memory of up to 8 clustered CTAs; select: 32 keys/thread

// Derived sizes of one problem.
struct Dims {
  int B, Hq, Hkv, g, n, d, seg, blk, k, n1, n2, r, es;  // es = element size in bytes
};

inline Dims make_dims(const cp_params& p) {
  Dims m;
  m.B = p.batch; m.Hq = p.n_q_heads; m.Hkv = p.n_kv_heads; m.g = p.n_q_heads / p.n_kv_heads;
  m.n = p.seq_len; m.d = p.head_dim; m.seg = p.segment_size; m.blk = p.block_size;
  m.k = p.budget_blocks;
  m.n1 = (p.seq_len + p.segment_size - 1) / p.segment_size;   // the last segment / block may be shorter
  m.n2 = (p.seq_len + p.block_size - 1) / p.block_size;
  m.r = p.segment_size / p.block_size; m.es = p.dtype == CP_F32 ? 4 : 2;
  return m;
}

// One sequence of a packed batch: where its S / idx / cnt arrays and its tokens start, and its length.
struct SeqSlot { int64_t s, idx, cnt, tok; int len; };
constexpr int kSeqsPerLaunch = 16;   // sequences whose descriptors travel in one launch's parameters

inline Dims seq_dims(const Dims& m, int len) {
  Dims x = m;
  x.n = len;
  x.n1 = (len + m.seg - 1) / m.seg;
  x.n2 = (len + m.blk - 1) / m.blk;
  return x;
}

// Workspace layout: [status 256 B][Qmax][Qmin][Kmax][Kmin][stats][kabs]: summaries in the input dtype;
// stats = the four log-sum-exps of every (head, segment) row, [B,Hq,n1,4] fp64; kabs = largest magnitude
// in each key block's summaries, [B,Hkv,n2] fp32.
struct WsLayout {
  size_t qmax, qmin, kmax, kmin, stats, kabs, total;
};
inline WsLayout ws_layout(const Dims& m) {
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  WsLayout w;
  size_t qs = up(size_t(m.B) * m.Hq * m.n1 * m.d * m.es);
  size_t ks = up(size_t(m.B) * m.Hkv * m.n2 * m.d * m.es);
  w.qmax = kStatusBytes; w.qmin = w.qmax + qs; w.kmax = w.qmin + qs; w.kmin = w.kmax + ks;
  w.stats = w.kmin + ks;
  w.kabs = w.stats + up(size_t(m.B) * m.Hq * m.n1 * 4 * sizeof(double));
  w.total = w.kabs + up(size_t(m.B) * m.Hkv * m.n2 * sizeof(float));
  return w;
}

// Query heads of a KV group that share a CTA of a score kernel.
inline int score_heads(const Dims& m) { return m.g % 4 == 0 ? 4 : (m.g % 2 == 0 ? 2 : 1); }
// Segments per CTA of the log-sum-exp kernel.  A CTA has 128 logit rows = 64 / U segments; on mid-sized problems fewer segments per CTA (rows left
// unused) put more SMs to work on the sweeps and the exact pass, which run per CTA one after the other.
inline int lse_segments(const Dims& m) {
  int segs = 64 / score_heads(m);
  const long long groups = (long long)m.B * m.Hkv * (m.g / score_heads(m));
  while (segs > 4 && groups * ((m.n1 + segs - 1) / segs) < 100) segs /= 2;
  return segs;
}

// Device status block.
struct DeviceStatus {
  int32_t code;     // cp_status, first error wins
  int32_t where;    // kernel-specific site id
  int32_t info[6];  // e.g. batch, head, segment, offending value
};

__device__ __forceinline__ void report(DeviceStatus* st, int code, int where, int a = 0, int b = 0,
                                       int c = 0, int d = 0) {
  if (st == nullptr) return;
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->where = where; st->info[0] = a; st->info[1] = b; st->info[2] = c; st->info[3] = d;
  }
}

// Kernel launchers (each returns a cp_status).
int launch_summarize(const cp_params& p, const Dims& m, const void* Q, const void* K, char* ws,
                     cudaStream_t s);
// the same for several sequences of a packed batch, each with a workspace of its own (ws[i])
int launch_summarize_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, char* const* ws, int n_seqs, const void* Q,
                          const void* K, cudaStream_t s);
int launch_score_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, char* const* ws, int n_seqs, const double* S_prev,
                      double* S_out, cudaStream_t s);      // sequences that score_is_split says no to
int launch_select_seqs(const cp_params& p, const Dims& m, const SeqSlot* slots, int n_seqs, const double* S, int32_t* idx, int32_t* cnt,
                       cudaStream_t s);
bool score_is_split(const cp_params& p, const Dims& m);    // the scores take the two-kernel path
int launch_score(const cp_params& p, const Dims& m, char* ws, const double* S_prev,
                 double* S_out, cudaStream_t s);
int launch_lse(const cp_params& p, const Dims& m, char* ws, cudaStream_t s);   // stats region of ws <- row log-sum-exps
int launch_score_generic(const cp_params& p, const Dims& m, const char* ws, const double* S_prev,
                         double* S_out, double* stats_out, cudaStream_t s);
int launch_select(const cp_params& p, const Dims& m, const double* S, int32_t* idx, int32_t* cnt,
                  cudaStream_t s, int past_fixed = -1);
int launch_attention_simt(const cp_params& p, const Dims& m, const void* Q, const void* K,
                          const void* V, const int32_t* idx, const int32_t* cnt, void* O, float* lse,
                          DeviceStatus* st, bool dense, cudaStream_t s);
int launch_attention_sm100(const cp_params& p, const Dims& m, const void* Q, const void* K,
                           const void* V, const int32_t* idx, const int32_t* cnt, void* O,
                           float* lse, DeviceStatus* st, bool dense, cudaStream_t s);
int launch_attention_sm100_varlen(const cp_params& p, const Dims& m, const SeqSlot* slots, int n_seqs, const void* Q, const void* K,
                                  const void* V, const int32_t* idx, const int32_t* cnt, void* O, float* lse, DeviceStatus* st,
                                  cudaStream_t s);
bool sm100_path_applies(const cp_params& p, const Dims& m);
int launch_project(const cp_params& p, const Dims& m, const void* X, const void* Wq, const void* Wk, const void* Wv,
                   const float* cosT, const float* sinT, int d_model, void* Q, void* K, void* V, char* ws, cudaStream_t st);

int launch_decode_score(const cp_params& p, const Dims& m, const void* q_last, const void* K, double* S_out, char* ws, cudaStream_t st);
bool decode_path_applies(const Dims& m);

// Programmatic dependent launch: a kernel starts while its predecessor drains, if that one calls pdl_trigger (those of the estimate, the
// selection, decoding and SIMT attention do; the projection and tensor-core attention don't, and have no successor before their end).  Every thread of such a kernel
// calls pdl_wait before it touches global memory (the predecessor has then finished and its writes are visible, so nothing else
// about stream order changes); pdl_trigger lets the successor start its own way to that point.  The pointers named in pdl_wait
// pass through it, so that no read-only load through them (__ldg, const __restrict__) can be scheduled before the wait.
template <typename P> __device__ __forceinline__ void asm_launder(P& ptr) { asm volatile("" : "+l"(ptr) :: "memory"); }
template <typename... P>
__device__ __forceinline__ void pdl_wait(P&... ptrs) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  (asm_launder(ptrs), ...);
}
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
int launch_pdl_cluster(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, unsigned cluster_x, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster_x; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster_x > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, P(args)...);
  const cudaError_t last = cudaGetLastError();
  return e == cudaSuccess && last == cudaSuccess ? CP_OK : CP_ERR_CUDA;
}
template <typename... P, typename... A>
int launch_pdl(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, const A&... args) {
  return launch_pdl_cluster(kern, grid, block, smem, 1, st, args...);
}

inline int check_launch() { return cudaGetLastError() == cudaSuccess ? CP_OK : CP_ERR_CUDA; }

}  // namespace cp
