// Internal declarations shared by the translation units of liblasdf.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/las.h"

#define LAS_MAX_FRAG 64
#define LAS_MAX_ACT 96  // total active orbitals handled by the per-L kernel (3a^2 doubles of smem)

// Device status word codes (first error wins; see las_status).
#define LAS_DEV_OK 0

#define LAS_CUDA_TRY(expr)                               \
  do {                                                   \
    cudaError_t e_ = (expr);                             \
    if (e_ != cudaSuccess) {                             \
      las_record_cuda_error(e_, #expr, __FILE__, __LINE__); \
      return LAS_ERR_CUDA;                               \
    }                                                    \
  } while (0)

void las_record_cuda_error(cudaError_t e, const char* what, const char* file, int line);

// Process-wide count of kernels this library has launched (diagnostics).
void las_count_launch(long k = 1);

// Programmatic dependent launches.  A kernel launched by launch_chained may start while the launch
// before it in the stream still runs: its blocks are placed as soon as all blocks of that one have
// begun, and wait in pdl_wait until it has completed and its writes are visible.  Every kernel
// launched this way calls pdl_wait (or pdl_begin) in all threads before it touches global memory,
// so completion is transitive along a chain.  An evaluation of a small problem is 16 launches of a
// few microseconds each, and this hides their launch latency and set-up (48 orbitals: 125 -> 104 us).
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
  pdl_trigger();
  pdl_wait();
}
// Launches of this thread are chained while a ChainScope of an uncaptured stream is alive (under
// stream capture they are ordinary launches).
extern thread_local bool g_chain_launches;
struct ChainScope {
  bool saved;
  explicit ChainScope(cudaStream_t s) : saved(g_chain_launches) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    g_chain_launches =
        cudaStreamIsCapturing(s, &st) == cudaSuccess && st == cudaStreamCaptureStatusNone;
  }
  ~ChainScope() { g_chain_launches = saved; }
  ChainScope(const ChainScope&) = delete;
  ChainScope& operator=(const ChainScope&) = delete;
};
// kern<<<grid, block, smem, s>>>(args...); errors are left to cudaGetLastError as with <<<>>>
template <class... P, class... A>
void launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                    A... args) {
  if (!g_chain_launches) {
    kern<<<grid, block, smem, s>>>(P(args)...);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// Fragment description in constant-size form (passed by value to kernels).
struct FragInfo {
  int nfrag;
  int ncore;
  int nact;                      // total active orbitals a
  int off[LAS_MAX_FRAG + 1];     // active offsets (relative to the first active orbital)
  long dm1_off[LAS_MAX_FRAG];    // offset of fragment K in dm1s (doubles)
  long dm2_off[LAS_MAX_FRAG];    // offset of fragment K in dm2 (doubles)
};

// ------------------------------------------------------------------------------------------
// Generic FP64 GEMM on DMMA (mma.sync.m16n8k4.f64):  C[b](m,n) (+)= alpha * sum_k A[b](m,k) B[b](k,n)
// (gemm_f64.cuh).  Operands are read through small loader objects so that packed-symmetric B,
// transposed views and batched/strided layouts share one kernel.
// ------------------------------------------------------------------------------------------
struct StridedA {  // element (b, m, k) = p[b*sb + m*sm + k*sk]
  const double* p;
  long sb, sm, sk;
  __device__ __forceinline__ double operator()(int b, int m, int k) const {
    return p[(long)b * sb + (long)m * sm + (long)k * sk];
  }
};

// Element (b, mu, nu) of the symmetric matrix b^L (L = l0 + b) stored packed lower-triangular.
struct PackedSymA {
  const double* Bp;
  long npair;
  long l0;
  __device__ __forceinline__ double operator()(int b, int mu, int nu) const {
    long hi = mu > nu ? mu : nu, lo = mu > nu ? nu : mu;
    return Bp[(l0 + b) * npair + hi * (hi + 1) / 2 + lo];
  }
};

struct StridedC {  // C[b*sb + m*sm + n*sn] (=|+=) alpha * acc
  double* p;
  long sb, sm, sn;
  double alpha;
  int accumulate;
  __device__ __forceinline__ void operator()(int b, int m, int n, double v) const {
    double* q = p + (long)b * sb + (long)m * sm + (long)n * sn;
    *q = accumulate ? (*q + alpha * v) : alpha * v;
  }
};

// Small helpers implemented in las_kernels.cu
// Cocc[n][op] = the first o columns of C (zero padding); with dm2 also the pair-transposed
// fragment 2-RDMs dm2t that launch_per_aux reads
void launch_pack_cocc(const double* C, int n, int nmo, int o, int op, double* Cocc,
                      cudaStream_t s, const double* dm2 = nullptr, const FragInfo* fi = nullptr,
                      double* dm2t = nullptr);
las_status per_aux_prepare();
// CT[k][mu] = Cocc[mu][k] for k < r (Cocc is n x op)
void launch_transpose_cols(const double* Cocc, int n, int op, int r, double* CT, cudaStream_t s);
// vc[b] (+)= sgn sum_{k<r} sum_mu Ht[(b*r + k)*n + mu] * CT[k*n + mu], b < nL (fixed summation
// order); and mx[mu] = max(mx[mu], max_{b,k} |Ht|) as bit patterns.  Either of vc, mx may be null.
void launch_trace_ht(const double* Ht, const double* CT, int nL, int r, int n, double* vc,
                     double sgn, int accumulate, unsigned long long* mx, cudaStream_t s);
// W_L of every aux row, and eps, vc, va.  gexp == nullptr: W[L][p][q]; otherwise W is written as
// Wt[q][L*op + p] * 2^gexp[L*op + p]
void launch_per_aux(const double* T, int nL, int op, const double* dm1s, const double* dm2t,
                    const FragInfo& fi, double* W, double* eps, double* vc, double* va,
                    int with_grad, const int* gexp, cudaStream_t s);
// K = scale * (its lower triangle, mirrored)
void launch_mirror_lower(double* K, int n, double scale, cudaStream_t s);
// out[q][k] = Wt[q][k] * 2^(g1[k] - g0[k]) for k < wld, q < rows: Wt scaled by 2^g1 instead of 2^g0
void launch_rescale_w(const double* Wt, long wld, int rows, const int* g0, const int* g1,
                      double* out, cudaStream_t s);
// dT[L] = X[L] + X[L]^T for L < nL (op x op each)
void launch_sym_add(const double* X, int nL, int op, double* dT, cudaStream_t s);
// Columns of each sign of w0 (idx, then idx + o: w > 0, w < 0) and of w1 (idx + 2 o, idx + 3 o) in
// order and their counts[4], then the packed factor of one sign
void launch_sign_split(const double* w0, int r0, const double* w1, int r1, int o, int* idx,
                       int* counts, cudaStream_t s);
void launch_pack_weighted(const double* Cx, const double* w, const int* idx, int cnt,
                          double sign, int n, int r, int op, double* Cocc, cudaStream_t s);
// out (+)= scale sum_k part[k*count ...] in order of k; with cols < ld the values are rows of
// `cols` that land `ld` apart in out
void launch_reduce_partials(const double* part, int nsplit, long count, double* out,
                            int accumulate, cudaStream_t s, long cols = 0, long ld = 0,
                            double scale = 1.0);
void launch_assemble_grad(const double* Out, const double* hC, const double* dm1s,
                          const FragInfo& fi, int n, int nmo, int op, double* G,
                          cudaStream_t s);
// *E = one-electron energy of h (hC = h C_occ) + sum_L eps_L; e1: E1_BLOCKS doubles of scratch; with
// G also launch_assemble_grad, in the same launch as the energy's sum
#define E1_BLOCKS 256
void launch_energy(const double* eps, int X, const double* Cocc, const double* hC, int n, int op,
                   const double* dm1s, const FragInfo& fi, double* e1, double* E, cudaStream_t s,
                   const double* Out = nullptr, int nmo = 0, double* G = nullptr);
void launch_antisym(const double* M, int nmo, int o, int op, double* g, cudaStream_t s);
// Jp[z][npair], z < parts: partial sums over parts of the auxiliary index (coulomb_parts: how many)
int coulomb_parts(long npair, int X, int sms);
void launch_coulomb_packed(const double* Bp, const double* vc, int X, long npair, int parts,
                           double* Jp, cudaStream_t s);
// J = scale * the symmetric matrix of the packed lower triangle sum_z Jp[z]
void launch_unpack_sym(const double* Jp, int parts, int n, double scale, double* J,
                       cudaStream_t s);
// va = J - Ka, vb = J - Kb from the packed J and the lower triangles of Ka, Kb
void launch_veff_combine(const double* Jp, int parts, const double* Ka, const double* Kb, int n,
                         double* va, double* vb, cudaStream_t s);
// Lmu[L][mu][u] = Ht[L][u][mu] for L < nL, u < a (at most LAS_MAX_ACT)
void launch_transpose_ht(const double* Ht, int nL, int n, int a, double* Lmu, cudaStream_t s);
