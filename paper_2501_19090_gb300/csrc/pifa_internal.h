// pifa_internal.h -- declarations shared by the host API (api.cpp) and the kernel files (*.cu).
// Not installed; the public interface is include/pifa.h.
#ifndef PIFA_INTERNAL_H_
#define PIFA_INTERNAL_H_

#include <stdint.h>

#include <cuda.h>
#include <cuda_runtime.h>

// ---- error reporting (api.cpp) ---------------------------------------------------------------
void pifa_clear_error();
int pifa_fail(int status, const char* msg);                       // records msg, returns status
int pifa_fail_cuda(const char* where, cudaError_t err);           // PIFA_ERR_CUDA with detail

// Device status word of the current device (api.cpp). Kernels latch the first error into it
// with atomicCAS(word, 0, code).
int* pifa_status_word(cudaError_t* err);

// Default bound of every device-side wait, nanoseconds (env PIFA_WAIT_TIMEOUT_NS overrides).
uint64_t pifa_wait_timeout_ns();

// Kernels this library has enqueued (status.cu): every launch site calls pifa_count_launch() once
// per successful launch; pifa_launch_count() reads the total.
void pifa_count_launch();

// SMs of the current device (status.cu); 1 if the query fails, which the next call makes again.
int pifa_sm_count();

#ifdef __CUDACC__
#include <utility>
// cudaLaunchKernelEx, counted.
template <typename... K, typename... A>
inline cudaError_t pifa_launch_ex(const cudaLaunchConfig_t* cfg, void (*kernel)(K...), A&&... args) {
  const cudaError_t e = cudaLaunchKernelEx(cfg, kernel, std::forward<A>(args)...);
  if (e == cudaSuccess) pifa_count_launch();
  return e;
}
#endif

// Shape of one forward call after validation (element counts and pitches).
struct PifaShape {
  int64_t T, m, n, r;
  int64_t ldx, ldwp, ldc, ldy;
  int c_dtype;  // PIFA_DTYPE_BF16 or PIFA_DTYPE_FP16 (storage type of C)
  // G layers of one shape sharing X (pifa_forward_grouped): W_p holds G r rows, C G (m - r) rows,
  // Y G m columns (the pivot / non-pivot indices are absolute columns of Y), y_p G r columns; the
  // non-pivot rows of group g read y_p's columns [g r, (g + 1) r). G > 1 needs (m - r) % 128 == 0
  // and r % 8 == 0, so that no tile spans two groups and every group's y_p columns start 16-byte
  // aligned.
  int64_t groups = 1;
};

// The first kWorkspaceReserve bytes of every workspace are reserved for library state (no kernel
// of this version uses them); per-call scratch starts after them.
constexpr int64_t kWorkspaceReserve = 256;

struct PifaPointers {
  const void* X;
  const void* Wp;
  const void* C;
  const int32_t* piv;
  const int32_t* nonpiv;
  void* Y;
  void* ws;           // per-call scratch (workspace + kWorkspaceReserve)
  int64_t ws_bytes;   // bytes available at ws
};

// Byte span [lo, hi) of a row-major matrix (rows x cols used elements, pitch ld, elem bytes);
// empty for a null base or no rows/columns. Used to reject outputs that overlap inputs.
struct PifaSpan {
  uintptr_t lo, hi;
};
inline PifaSpan pifa_span(const void* base, int64_t rows, int64_t cols, int64_t ld, int64_t elem) {
  const uintptr_t b = reinterpret_cast<uintptr_t>(base);
  if (!base || rows <= 0 || cols <= 0) return {0, 0};
  return {b, b + (uintptr_t)(((rows - 1) * ld + cols) * elem)};
}
inline bool pifa_spans_overlap(PifaSpan a, PifaSpan b) {
  return a.lo < a.hi && b.lo < b.hi && a.lo < b.hi && b.lo < a.hi;
}

// ---- decode (decode.cu) ----------------------------------------------------------------------
int64_t decode_workspace_bytes(const PifaShape& s);
int launch_decode(const PifaShape& s, const PifaPointers& p, int* status, cudaStream_t stream);

// ---- decode on the tensor cores, split over K (decode_tc.cu) ------------------------------------
// One decode phase D = A B^T (A: R x K weight rows, B: T <= 128 token rows of K columns, NB =
// planes 1 or 2) as a split-K tcgen05 kernel: row blocks in clusters that add up their K-slices
// and write Y[t, cols[j]] (and, for phase 1, the y_p hi/lo planes) themselves, or, for phases of
// more row blocks than the grid holds, balanced ranges writing fp32 partial sums P and a reduction.
struct DecodeTcPhase {
  const void* A;
  int64_t lda, R, K;
  int dtype;            // storage type of A and B (PIFA_DTYPE_*)
  const void* B0;       // first (or only) B plane: T x bcols, pitch ldb
  const void* B1;       // second plane (planes == 2)
  int64_t ldb, bcols, T;
  int planes;
  int64_t gsz, goff;    // grouped layers: rows per group and B columns per group (0: one layer)
  bool mma_f16;         // A and B fp16 (else bf16)
  bool split_f16;       // phase 1: split y_p into fp16 hi/lo (else bf16)
  float* P;             // partial sums, decode_tc_partial_bytes(R, K, T, planes) bytes
  const int32_t* cols;  // output column of each weight row
  int64_t m;            // columns of Y (index bound)
  void* Y;
  int64_t ldy;
  uint16_t* yph;        // phase 1 with m > r: y_p planes (T x ldyp), else null
  uint16_t* ypl;
  int64_t ldyp;
};
int64_t decode_tc_partial_bytes(int64_t R, int64_t K, int64_t T, int NB);
int launch_decode_tc(const DecodeTcPhase& ph, int* status, uint64_t timeout_ns, cudaStream_t stream);

// ---- general tensor-core contraction (gemm_tc.cu) ------------------------------------------------
// D (M x N) = alpha A B^T (+ addend), bf16 operands, fp32 accumulation. A is M x K, B is N x K; each
// is K-major (a_mn = false: element (i, k) at [i * ld + k]) or MN-major (true: at [k * ld + i]).
// out_mode 0: D bf16; 1: D fp32; 2: D fp32 += result; 3: D = bf16 hi, D2 = bf16 lo of the result;
// 4: D = one bit per element, uint32 words of 32 columns, ldd words a row: whether the result S is
// neither zero nor at least alpha sqrt(k), k the element's terms (GemmF64's check, see `tri`).
// A2 / B2 (optional, A's / B's layout and pitch): a second K pass with A2 for A and / or B2 for B,
// D = (A + A2) B^T or A (B + B2)^T. Optional addend (out_mode 0 and 3): D[i][j] += add[i * ldadd + j]
// (bf16). Pointers 16-byte aligned, leading dimensions multiples of 8 elements (the caller checks).
struct GemmTc {
  int64_t M, N, K;
  const void* A;
  int64_t lda;
  bool a_mn;
  const void* B;
  int64_t ldb;
  bool b_mn;
  void* D;
  int64_t ldd;
  int out_mode;
  float alpha;
  const void* add;
  int64_t ldadd;
  const void* A2 = nullptr;
  const void* B2 = nullptr;
  void* D2 = nullptr;
  bool upper = false;    // M == N: skip 128 x 128 blocks wholly below the diagonal (a symmetric product)
  int tri = 0, k0 = 0, k1 = 0;  // out_mode 4: the columns [k0, k1) of a contraction with GemmF64's zeros `tri`
};
// Up to three independent products in one launch.
int gemm_tc_group(const GemmTc* gs, int n, int* status, uint64_t timeout_ns, cudaStream_t stream);

// ---- float64 products (compress_gpu.cu, gemm_f64_tc.cu) -------------------------------------------
// C[i][ccol(j)] = beta C + alpha sum_k A(i, k) B(k, j), with
//   A(i, k) = A[arow(i) * sa_i + k * sa_k],  arow(i) = aidx ? aidx[i] : i
//   B(k, j) = B[k * sb_k + j * sb_j]
//   C at C[i * ldc + (cidx ? cidx[j] : j)]
// and, on the CUDA cores, a batch index z (blockIdx.z) offsetting A, B and C by za, zb, zc elements.
// `tri` (bits): 1 B(k, j) = 0 for k < j, 2 B(k, j) = 0 for k > j, 4 A(i, k) = 0 for k < i; the k loop
// skips those zeros (k counts from kbase on). `lower`: only the tiles that hold some i >= j are computed.
// `normwise`: an error of a small multiple of 2^-62 sqrt(K) max_k |A(i, k)| max_k |B(k, j)| in element (i, j)
// is as good as float64's for the caller (see gemm_f64_split).
struct GemmF64 {
  int M, N, K;
  const double* A;
  const int32_t* aidx;
  int64_t sa_i, sa_k;
  const double* B;
  int64_t sb_k, sb_j;
  double* C;
  const int32_t* cidx;
  int64_t ldc;
  double alpha, beta;
  int tri;
  int64_t za, zb, zc;
  int lower;
  int normwise;
  int kbase;
};
// The same on the tensor cores by exact slices (no batch), in `bytes` of scratch:
// whether that form takes the product, and the product. slices > 1: the contraction cut into that many
// partial results, zc elements apart, each added to or stored in its own C, for the caller to add up
// (products of few tiles).
bool gemm_f64_split_fits(const GemmF64& p, int64_t bytes);
int gemm_f64_split(const GemmF64& p, void* scratch, int64_t bytes, cudaStream_t stream, int slices = 1, int64_t zc = 0);
// The elements of p whose bit is set in `mask` (uint32 words of 32 columns, `words` a row), on the CUDA cores.
int gemm_f64_flagged(const GemmF64& p, const uint32_t* mask, int words, cudaStream_t stream);

// ---- prefill (prefill.cu) --------------------------------------------------------------------
int64_t prefill_split_workspace_bytes(const PifaShape& s);
int launch_prefill_split(const PifaShape& s, const PifaPointers& p, int* status, uint64_t timeout_ns,
                         cudaStream_t stream);

// ---- TMA descriptors (api.cpp) ---------------------------------------------------------------
// 2-D tensor map over a row-major (rows x cols) matrix of 2-byte elements (bf16 or fp16, a
// PIFA_DTYPE_*) with row pitch `ld` elements; box of box_cols x box_rows elements, 128-byte
// swizzle, zero fill outside the matrix.
int make_tmap_2d(CUtensorMap* map, int dtype, const void* base, int64_t rows, int64_t cols, int64_t ld,
                 uint32_t box_cols, uint32_t box_rows);

#endif  // PIFA_INTERNAL_H_
