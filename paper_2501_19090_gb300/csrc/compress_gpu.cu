// compress_gpu.cu -- the float64 set-up steps on the GPU: pifa_compress_device (Algorithm 1,
// Sec. 3.2) and pifa_m_reconstruct (the two solves of the M reconstruction, Sec. 4, at the end).
//
// Route (all device-resident, float64; the caller's workspace holds every temporary):
//   1. G = V^T V (r x r) and its Cholesky factor L (G = L L^T). Then Z = U L (m x r) has the row
//      inner products of W' = U V^T: z_i . z_j = u_i G u_j^T = w_i . w_j, so QR with column
//      pivoting on W'^T (Algorithm 1, step 1) selects the same rows when run on Z^T, whose columns
//      are r long instead of n.
//   2. r greedy Businger-Golub steps on the rows of Z: step k picks the unchosen row of largest
//      residual norm (norms recomputed from the reflected rows, no downdating; ties to the lowest
//      index), builds the Householder reflector that maps the pivot row's residual onto e_k, and
//      applies it to every unchosen row; on large layers, at first to the candidates of up to 64
//      steps only and then to the other rows in one product ("candidate blocks" below). After r steps a chosen row holds its column of
//      the triangular factor R (selection order) and every other row i holds c_i = Q^T z_i.
//   3. Eq. 2 in Z-space: Z_np = C Z_p, with Z_p = R^T Q^T and Z_np = Cmat Q^T (rows c_i), so
//      C = Cmat R^{-T} -- one GEMM against the explicit inverse of R (computed by doubling:
//      inverted 32 x 32 diagonal blocks, then off-diagonal blocks -A^{-1} B D^{-1} level by level).
//      Columns go from selection order to ascending I as they are written.
//   4. W_p = U[I, :] V^T (Eq. 1).
// Products of 2^20 multiply-adds and more run on the tensor cores by exact slices (gemm_f64_tc.cu), the
// elements for which those are less exact than float64 arithmetic excepted (gemm_f64_masked);
// small ones, the panels of the Cholesky factorisation and the greedy steps run on the CUDA cores,
// bound by the float64 issue rate (about two multiply-adds per clock and SM). Measured against what
// this replaced (all products on the CUDA cores; Cholesky by rank-1 updates; every step over every
// row), 4096 x 4096, r = 2048: products 90.4, Cholesky 37.8 and steps 173 of 308 ms; now products
// with their slices and checks 16, Cholesky 2.2 and steps 38 of 59.6 ms. The M solves at m = n = 2048, r = 1024:
// 141.4 -> 11.7 ms. No kernel waits on another CTA.
#include <cmath>
#include <cstdio>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"
#include "recip.h"

namespace {

using namespace pifa;


// ---- float64 GEMM on the CUDA cores (GemmF64 in pifa_internal.h): small products ------------
// GT x GT output tiles, K step 16; 256 threads of (GT / 16)^2 outputs each. Tiles of 32 where those of
// 64 are fewer than the SMs, each bound by its SM's float64 pipe (a tile of 64 and K = 128: 130 us): the
// levels of a triangular inverse below 256, r = 1024 or 2048: 86 -> 25 us a launch.
constexpr int GK = 16;
constexpr int kSms = 152;
constexpr int kZeroBlock = 64;  // triangular operands: zeros are skipped in blocks of 64, whatever the tile

// Columns of the contraction that hold anything in the GT x GT tile at (i0, j0), of 0 .. K.
__device__ __forceinline__ void k_range(const GemmF64& p, int i0, int j0, int& kbeg, int& kend) {
  kbeg = 0;
  kend = p.K;
  const int ib = i0 / kZeroBlock * kZeroBlock, jb = j0 / kZeroBlock * kZeroBlock;
  if (p.tri & 1) kbeg = max(0, jb - p.kbase);
  if (p.tri & 4) kbeg = max(kbeg, ib - p.kbase);
  if (p.tri & 2) kend = min(p.K, jb + kZeroBlock - p.kbase);
}

// The tile's sums, one chain of multiply-adds per element, in the order of k: thread (tx, ty) of 16 x 16
// gets elements (i0 + ty + 16 u, j0 + tx + 16 v).
template <int GT>
__device__ __forceinline__ void tile_f64(const GemmF64& p, const double* A, const double* B, int i0, int j0,
                                         double (&acc)[GT / 16][GT / 16]) {
  constexpr int U = GT / 16;
  __shared__ double As[GK][GT + 1];
  __shared__ double Bs[GK][GT + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int kbeg, kend;
  k_range(p, i0, j0, kbeg, kend);
  for (int k0 = kbeg; k0 < kend; k0 += GK) {
    for (int e = threadIdx.x; e < GT * GK; e += 256) {
      const int ii = e % GT, kk = e / GT;  // consecutive threads: consecutive rows of the A tile
      const int i = i0 + ii, k = k0 + kk;
      double va = 0.0;
      if (i < p.M && k < p.K) {
        const int64_t row = p.aidx ? (int64_t)p.aidx[i] : (int64_t)i;
        va = A[row * p.sa_i + (int64_t)k * p.sa_k];
      }
      As[kk][ii] = va;
      const int jj = e % GT, j = j0 + jj;
      double vb = 0.0;
      if (j < p.N && k < p.K) vb = B[(int64_t)k * p.sb_k + (int64_t)j * p.sb_j];
      Bs[kk][jj] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      double a[U], b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u] = As[kk][ty + 16 * u];
        b[u] = Bs[kk][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void store_f64(const GemmF64& p, double* C, int i, int j, double sum) {
  double* c = C + (int64_t)i * p.ldc + (p.cidx ? (int64_t)p.cidx[j] : (int64_t)j);
  *c = (p.beta != 0.0 ? p.beta * *c : 0.0) + p.alpha * sum;
}

template <int GT>
__global__ void __launch_bounds__(256) gemm_f64(GemmF64 p) {
  constexpr int U = GT / 16;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.y * GT, j0 = blockIdx.x * GT;
  double* C = p.C + blockIdx.z * p.zc;
  if (p.lower && j0 > i0 + GT - 1) return;
  double acc[U][U] = {};
  tile_f64<GT>(p, p.A + blockIdx.z * p.za, p.B + blockIdx.z * p.zb, i0, j0, acc);
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      if (i < p.M && j < p.N) store_f64(p, C, i, j, acc[u][v]);
    }
}

// The flagged elements of a 32 x 32 tile per CTA: the tile's sums where many are flagged, else a thread per
// element with the same chain, so that an element's value does not depend on its neighbours' flags (equal
// rows keep equal values). Bound by the float64 pipe: a tile of K columns holds its SM for 512 K cycles,
// up to kFewFlags elements alone for 64 K.
constexpr int kFewFlags = 64;
__global__ void __launch_bounds__(256) gemm_f64_masked(GemmF64 p, const uint32_t* mask, int words) {
  __shared__ uint32_t s_mask[32];
  __shared__ int s_at[33];
  __shared__ uint16_t s_list[kFewFlags];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    // bits beyond N are zero, unless the product that writes the mask gave up a wait and left it as it was
    const uint32_t in = p.N - j0 < 32 ? (1u << (p.N - j0)) - 1u : 0xffffffffu;
    const uint32_t w = i0 + lane < p.M ? mask[(int64_t)(i0 + lane) * words + blockIdx.x] & in : 0u;
    s_mask[lane] = w;
    int at = __popc(w);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += x;
    }
    s_at[lane + 1] = at;
    if (lane == 0) s_at[0] = 0;
  }
  __syncthreads();
  const int n = s_at[32];
  if (n == 0) return;
  if (n > kFewFlags) {
    double acc[2][2] = {};
    tile_f64<32>(p, p.A, p.B, i0, j0, acc);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v)
        if (s_mask[ty + 16 * u] >> (tx + 16 * v) & 1u) store_f64(p, p.C, i0 + ty + 16 * u, j0 + tx + 16 * v, acc[u][v]);
    return;
  }
  if (threadIdx.x < 32) {
    int at = s_at[threadIdx.x];
    for (uint32_t w = s_mask[threadIdx.x]; w; w &= w - 1) s_list[at++] = (uint16_t)(threadIdx.x * 32 + __ffs(w) - 1);
  }
  __syncthreads();
  if ((int)threadIdx.x >= n) return;
  const int i = i0 + (s_list[threadIdx.x] >> 5), j = j0 + (s_list[threadIdx.x] & 31);
  int kbeg, kend;
  k_range(p, i0, j0, kbeg, kend);
  const double* a = p.A + (p.aidx ? (int64_t)p.aidx[i] : (int64_t)i) * p.sa_i;
  const double* b = p.B + (int64_t)j * p.sb_j;
  double sum = 0.0;
#pragma unroll 8
  for (int k = kbeg; k < kend; ++k) sum = fma(a[(int64_t)k * p.sa_k], b[(int64_t)k * p.sb_k], sum);
  store_f64(p, p.C, i, j, sum);
}

int run_gemm_f64(const GemmF64& p, int batch, cudaStream_t s) {
  if (p.M <= 0 || p.N <= 0 || batch <= 0) return PIFA_OK;
  const auto grid = [&](int gt) { return dim3((unsigned)((p.N + gt - 1) / gt), (unsigned)((p.M + gt - 1) / gt), (unsigned)batch); };
  const int64_t tiles = (int64_t)((p.N + 63) / 64) * ((p.M + 63) / 64) * batch;
  if (tiles < kSms) gemm_f64<32><<<grid(32), 256, 0, s>>>(p);
  else gemm_f64<64><<<grid(64), 256, 0, s>>>(p);
  pifa_count_launch();
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PIFA_OK : pifa_fail_cuda("compress: gemm launch", e);
}

// The same product by whichever form takes it: on the tensor cores by exact slices (gemm_f64_tc.cu)
// from 2^20 multiply-adds on, with the caller's free scratch for the sliced operands, else on the
// CUDA cores (one 64 x 64 tile of K = 128 keeps an SM's float64 pipe busy for about 130 us).
int run_product(const GemmF64& p, void* scratch, int64_t bytes, cudaStream_t s) {
  if (p.M <= 0 || p.N <= 0) return PIFA_OK;
  if (gemm_f64_split_fits(p, bytes)) return gemm_f64_split(p, scratch, bytes, s);
  return run_gemm_f64(p, 1, s);
}

// ---- Cholesky of G (r x r, pitch r, lower triangle used and overwritten) -------------------------
// Blocked, right-looking: panels of 128 columns, each 32 columns at a time (chol_panel, then
// chol_update for the rest of the panel), and the trailing matrix updated once per panel by a
// K = 128 product. The predecessor, one rank-1 update of the whole trailing matrix with a division
// per element and a launch per column, took 37.8 ms at r = 2048.
constexpr int CB = 32;    // columns per chol_panel
constexpr int CP = 128;   // columns per panel

constexpr int CR = 32;    // rows below the diagonal block per CTA of chol_panel

// Columns [j0, j0 + CB) of L. Every CTA factors the 32 x 32 diagonal block itself (as U D U^T with
// unit-lower U): the warp that holds column j + 1 finishes it first and takes its reciprocal while the
// other three update the rest, so that a column's critical path is one multiply-add, one reciprocal,
// one multiplication and one barrier. Then four lanes per row below it substitute that row. A
// non-positive pivot flags `bad` and leaves its column of L zero.
// Bound by the float64 pipe (one warp instruction per 64 cycles and scheduler). r = 2048: 45 -> 27 us
// against a division per column in every warp and a thread per row.
__global__ void __launch_bounds__(128) chol_panel(const double* G, double* L, int r, int j0, int* bad) {
  __shared__ double D[CB][CB + 1];  // the block; column l of its lower part ends as d_l U[:, l]
  __shared__ double U[CB][CB + 1];
  __shared__ double rd[CB], rs[CB];  // 1 / d_l and 1 / sqrt(d_l), 0 where d_l is not positive
  pdl_launch_dependents();
  pdl_wait_primary();
  const int nb = min(CB, r - j0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this lane's share of a row below: columns 4 u + lane % 4
  const int64_t i = (int64_t)j0 + CB + (int64_t)blockIdx.x * CR + (threadIdx.x >> 2);
  const int q = lane & 3;
  double y[CB / 4];
#pragma unroll
  for (int u = 0; u < CB / 4; ++u) y[u] = i < r ? G[i * r + j0 + 4 * u + q] : 0.0;
  for (int k = warp; k < CB; k += 4)
    D[k][lane] = (k < nb && lane < nb) ? G[(int64_t)(j0 + k) * r + j0 + lane] : (k == lane ? 1.0 : 0.0);
  __syncthreads();
  if (warp == 0) {
    const double d = D[0][0], inv = d > 0.0 ? recip(d) : 0.0;
    if (lane == 0) rd[0] = inv;
  }
  __syncthreads();
  for (int j = 0; j < CB; ++j) {
    const double f = D[lane][j] * rd[j];
    if (warp == (j & 3)) {  // column j + 1 and its reciprocal; it has a warp to itself
      U[lane][j] = f;
      if (j + 1 < CB) {
        const double x = fma(-f, D[j + 1][j], D[lane][j + 1]);
        if (lane >= j + 1) D[lane][j + 1] = x;
        const double d = __shfl_sync(0xffffffffu, x, j + 1), inv = d > 0.0 ? recip(d) : 0.0;
        if (lane == 0) rd[j + 1] = inv;
      }
    } else {
      const int w = (warp - j + 3) & 3;  // 0, 1, 2 among the others
      for (int l = j + 2 + w; l < CB; l += 3)
        if (lane >= l) D[lane][l] = fma(-f, D[l][j], D[lane][l]);
    }
    __syncthreads();
  }
  if (warp == 0) {
    const double d = D[lane][lane];
    rs[lane] = d > 0.0 ? 1.0 / sqrt(d) : 0.0;
    if (!(d > 0.0) && blockIdx.x == 0) atomicExch(bad, 1);
  }
#pragma unroll
  for (int l = 0; l < CB; ++l) {  // y_j -= y_l U_jl
    const double x = __shfl_sync(0xffffffffu, y[l / 4], (lane & ~3) | (l & 3));
#pragma unroll
    for (int u = l / 4; u < CB / 4; ++u)
      if (4 * u + q > l) y[u] = fma(-x, U[4 * u + q][l], y[u]);
  }
  __syncthreads();
  if (i < r) {
    double* o = L + i * r + j0;
#pragma unroll
    for (int u = 0; u < CB / 4; ++u) o[4 * u + q] = y[u] * rs[4 * u + q];
  }
  if (blockIdx.x == 0)
    for (int k = warp; k < nb; k += 4)
      if (lane <= k) L[(int64_t)(j0 + k) * r + j0 + lane] = D[k][lane] * rs[lane];
}

// G[i][l] -= sum over k in [j0, j0 + kn) of L[i][k] L[l][k] for l0 <= l < l1, i >= l (kn <= CB).
// 16 x 32 tiles, 256 threads, 2 rows of one column each: bound by the float64 pipe of the SM that has
// the most tiles (r = 2048: 22 -> 8.4 us against 64 x 32 tiles, fewer than SMs).
constexpr int CU = 16;
__global__ void __launch_bounds__(256) chol_update(double* G, const double* L, int r, int j0, int kn, int l0, int l1) {
  __shared__ double A[CU][CB + 1];
  __shared__ double B[CB][CB + 1];
  const int i0 = l0 + blockIdx.y * CU, c0 = l0 + blockIdx.x * 32;
  pdl_launch_dependents();
  pdl_wait_primary();
  if (c0 > i0 + CU - 1) return;  // wholly above the diagonal
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int u = warp; u < CU; u += 8) A[u][lane] = (i0 + u < r && lane < kn) ? L[(int64_t)(i0 + u) * r + j0 + lane] : 0.0;
  for (int u = warp; u < 32; u += 8) B[u][lane] = (c0 + u < l1 && lane < kn) ? L[(int64_t)(c0 + u) * r + j0 + lane] : 0.0;
  __syncthreads();
  double acc[CU / 8] = {};
#pragma unroll 8
  for (int k = 0; k < CB; ++k) {
    const double b = B[lane][k];
#pragma unroll
    for (int u = 0; u < CU / 8; ++u) acc[u] = fma(A[warp * (CU / 8) + u][k], b, acc[u]);
  }
  const int l = c0 + lane;
#pragma unroll
  for (int u = 0; u < CU / 8; ++u) {
    const int i = i0 + warp * (CU / 8) + u;
    if (i < r && l < l1 && i >= l) G[(int64_t)i * r + l] -= acc[u];
  }
}

// L (zeroed by the caller, pitch r) = the Cholesky factor of G; `scratch` for the sliced panels.
int cholesky(double* G, double* L, int64_t r, int* bad, void* scratch, int64_t bytes, cudaStream_t s) {
  const int ri = (int)r;
  cudaError_t e = cudaSuccess;
  // each launch under the tail of the one before (224 launches of the M solves at n = 2048: 11.7 -> 11.3 ms)
  auto launch = [&](auto kernel, dim3 grid, int threads, auto... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (e == cudaSuccess) e = pifa_launch_ex(&cfg, kernel, args...);
  };
  for (int p0 = 0; p0 < ri; p0 += CP) {
    const int p1 = p0 + CP < ri ? p0 + CP : ri;
    GemmF64 t = {};  // the trailing update: G[p1:, p1:] -= L[p1:, p0:p1] L[p1:, p0:p1]^T
    t.M = t.N = ri - p1; t.K = p1 - p0;
    t.A = t.B = L + (int64_t)p1 * r + p0; t.sa_i = t.sb_j = r; t.sa_k = t.sb_k = 1;
    t.C = G + (int64_t)p1 * r + p1; t.ldc = r; t.alpha = -1.0; t.beta = 1.0; t.lower = 1;
    const bool split = t.M > 0 && gemm_f64_split_fits(t, bytes);
    for (int j0 = p0; j0 < p1; j0 += CB) {
      const int below = ri - j0 - CB;
      launch(chol_panel, dim3(below > 0 ? (unsigned)((below + CR - 1) / CR) : 1u), 128, (const double*)G, L, ri, j0, bad);
      const int l1 = split ? p1 : ri;  // without the product, 32 columns at a time over everything
      const int l0 = j0 + CB;
      if (l0 < l1)
        launch(chol_update, dim3((unsigned)((l1 - l0 + 31) / 32), (unsigned)((ri - l0 + CU - 1) / CU)), 256, G, (const double*)L,
               ri, j0, ri - j0 < CB ? ri - j0 : CB, l0, l1);
    }
    if (e != cudaSuccess) return pifa_fail_cuda("cholesky: launch", e);
    if (split) {
      const int st = gemm_f64_split(t, scratch, bytes, s);
      if (st != PIFA_OK) return st;
    }
  }
  return PIFA_OK;
}

// ---- greedy pivoted QR on the rows of Z -------------------------------------------------------
// Best and runner-up residual norms (squared, as float64 bit patterns: non-negative values order
// like their bits) with their rows, and the best one's slot in the list of unchosen rows; larger
// norm first, then the lower row: the selection rule of Algorithm 1, step 1 with ties to the lowest
// index.
struct Top2 {
  unsigned long long v1, v2;
  int i1, i2, s1;
};

__device__ __forceinline__ void top2_add(Top2& t, unsigned long long v, int i, int s) {
  if (i < 0) return;
  if (t.i1 < 0 || v > t.v1 || (v == t.v1 && i < t.i1)) {
    t.v2 = t.v1;
    t.i2 = t.i1;
    t.v1 = v;
    t.i1 = i;
    t.s1 = s;
  } else if (t.i2 < 0 || v > t.v2 || (v == t.v2 && i < t.i2)) {
    t.v2 = v;
    t.i2 = i;
  }
}

// The key of a squared norm; a NaN (a row of U that holds one) ranks below every number.
__device__ __forceinline__ unsigned long long norm_key(double v) {
  return v >= 0.0 ? (unsigned long long)__double_as_longlong(v) : 0ull;
}

__device__ __forceinline__ Top2 top2_empty() { return Top2{0ull, 0ull, -1, -1, -1}; }

__device__ __forceinline__ void top2_merge(Top2& a, const Top2& b) {
  top2_add(a, b.v1, b.i1, b.s1);
  top2_add(a, b.v2, b.i2, -1);  // never a's best: b's best is in front of it
}

__device__ Top2 warp_top2(Top2 t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Top2 u;
    u.v1 = __shfl_xor_sync(0xffffffffu, t.v1, o);
    u.v2 = __shfl_xor_sync(0xffffffffu, t.v2, o);
    u.i1 = __shfl_xor_sync(0xffffffffu, t.i1, o);
    u.i2 = __shfl_xor_sync(0xffffffffu, t.i2, o);
    u.s1 = __shfl_xor_sync(0xffffffffu, t.s1, o);
    top2_merge(t, u);
  }
  return t;
}

// Block-wide Top2 (at most 16 warps): every thread gets the block's result.
__device__ Top2 block_top2(Top2 t) {
  __shared__ Top2 sw[16];
  t = warp_top2(t);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sw[w] = t;
  __syncthreads();
  return warp_top2(lane < (int)(blockDim.x >> 5) ? sw[lane] : top2_empty());
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int kGreedyBlocks = 152;  // one per SM

struct Greedy {
  double* Z;        // m x r, row-major
  int m, r;
  int32_t* sel;     // m flags: chosen in an earlier step
  int32_t* act;     // the unchosen rows: m - k of them before step k
  Top2* blk;        // 2 x nblk per-block results (ping-pong by step parity)
  int nblk;
  int32_t* order;   // r: row chosen at step k
  double* rdiag;    // r: R_kk of the pivoted QR
  double* gap;      // r: (best - runner-up) / best of the residual norms at step k
  struct GreedyCtl* ctl;
  double* tau;      // r: the reflectors' tau (candidate blocks only, else null)
};

// The rows that a run of steps works on, set by greedy_select.
struct GreedyCtl {
  int stop, k_end;           // set by the step that could not be sure of its pivot
  int count;                 // rows in the list at the run's first step
  int all;                   // 1: every unchosen row is in the list
  unsigned long long theta;  // else: no other row's squared norm exceeded this at the run's first step
};

// Initial squared row norms of Z, each block's best two, and the list of all rows (the exhaustive
// steps from 0 on, without a norm's scratch per row).
__global__ void __launch_bounds__(256) greedy_init(Greedy g) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Top2 t = top2_empty();
  for (int i = blockIdx.x * 8 + warp; i < g.m; i += gridDim.x * 8) {
    const double* z = g.Z + (int64_t)i * g.r;
    double s = 0.0;
    for (int c = lane; c < g.r; c += 32) s = fma(z[c], z[c], s);
    s = warp_sum(s);
    if (lane == 0) {
      top2_add(t, norm_key(s), i, i);
      g.act[i] = i;
    }
  }
  t = block_top2(t);
  if (threadIdx.x == 0) g.blk[blockIdx.x] = t;
  if (blockIdx.x == 0 && threadIdx.x == 0) *g.ctl = GreedyCtl{0, 0, g.m, 1, 0ull};
}

// Squared residual norms (coordinates k..r-1) of the unchosen rows; -1 marks a chosen one.
__global__ void __launch_bounds__(256) greedy_norms(Greedy g, int k, double* norms) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = blockIdx.x * 8 + warp; i < g.m; i += gridDim.x * 8) {
    const double* z = g.Z + (int64_t)i * g.r;
    double s0 = 0.0, s1 = 0.0;
    if (!g.sel[i]) {
      int c = k + lane;
      for (; c + 32 < g.r; c += 64) {
        s0 = fma(z[c], z[c], s0);
        s1 = fma(z[c + 32], z[c + 32], s1);
      }
      if (c < g.r) s0 = fma(z[c], z[c], s0);
    }
    s0 = warp_sum(s0 + s1);
    if (lane == 0) norms[i] = g.sel[i] ? -1.0 : s0;
  }
}

// The list for the steps from k on and their first best two: the rows of the `want` or somewhat fewer
// largest norms (a threshold found by bisection; in_list marks them), or, with want = 0 or where
// ties leave fewer than a quarter of them above any threshold, all unchosen rows. One block of 1024.
// The norms are compared as integers (their bits; -1 for a chosen row, 0 for a NaN), the first 4096 of
// them kept in registers: float64 comparisons of values read again at each step took 35 us, these 17 (m = 4096).
__global__ void __launch_bounds__(1024) greedy_select(Greedy g, int k, const double* norms, int want, uint8_t* in_list) {
  __shared__ int s_n[32];
  __shared__ long long s_m[32];
  __shared__ Top2 s_t[32];
  __shared__ int s_count;
  constexpr int HELD = 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto key = [&](int i) {
    const long long b = __double_as_longlong(norms[i]), a = b & 0x7fffffffffffffffll;
    return b == (long long)0xbff0000000000000ull ? -1ll : a > 0x7ff0000000000000ll ? 0ll : a;  // -1.0: chosen
  };
  long long held[HELD], mx = 0;
#pragma unroll
  for (int u = 0; u < HELD; ++u) {
    const int i = threadIdx.x + 1024 * u;
    held[u] = i < g.m ? key(i) : -1ll;
    mx = max(mx, held[u]);
  }
  for (int i = threadIdx.x + 1024 * HELD; i < g.m; i += 1024) mx = max(mx, key(i));
  auto count_above = [&](long long th) {
    int n = 0;
#pragma unroll
    for (int u = 0; u < HELD; ++u) n += held[u] > th ? 1 : 0;
    for (int i = threadIdx.x + 1024 * HELD; i < g.m; i += 1024) n += key(i) > th ? 1 : 0;
    n = __reduce_add_sync(0xffffffffu, n);
    __syncthreads();
    if (lane == 0) s_n[warp] = n;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, s_n[lane]);
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, (long long)__shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_m[warp] = mx;
  __syncthreads();
  mx = s_m[lane];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, (long long)__shfl_xor_sync(0xffffffffu, mx, o));
  // count above -1: all unchosen rows; above hi: none. Midpoints of the values, not of their bits.
  long long lo = -1, hi = mx;
  bool all = want == 0 || count_above(-1) <= 2 * want;
  long long th = lo;
  for (int it = 0; it < 48 && !all; ++it) {
    const double a = lo < 0 ? 0.0 : __longlong_as_double(lo);
    const long long mid = __double_as_longlong(0.5 * (a + __longlong_as_double(hi)));
    const int n = count_above(mid);
    if (n > want) {
      lo = mid;
    } else {
      hi = mid;
      th = mid;
      if (n >= want - want / 10) break;
    }
  }
  if (!all && (th < 0 || count_above(th) < want / 4)) all = true;
  if (all) th = -1;
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  Top2 t = top2_empty();
  for (int i0 = 0; i0 < g.m; i0 += 1024) {
    const int i = i0 + (int)threadIdx.x;
    const long long ki = i < g.m ? key(i) : -1ll;
    const bool in = ki > th;
    if (in_list && i < g.m) in_list[i] = in ? 1 : 0;
    const unsigned ballot = __ballot_sync(0xffffffffu, in);
    int at = 0;
    if (lane == 0 && ballot) at = atomicAdd(&s_count, __popc(ballot));  // the list's order changes no result
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(ballot & ((1u << lane) - 1u));
    if (in) {
      g.act[at] = i;
      top2_add(t, (unsigned long long)ki, i, at);
    }
  }
  t = warp_top2(t);
  if (lane == 0) s_t[warp] = t;
  __syncthreads();
  t = warp_top2(s_t[lane]);
  for (int b = threadIdx.x; b < g.nblk; b += 1024) g.blk[(k & 1) * g.nblk + b] = b == 0 ? t : top2_empty();
  if (threadIdx.x == 0) {
    g.ctl->stop = 0;
    g.ctl->k_end = 0;
    g.ctl->count = s_count;
    g.ctl->all = all ? 1 : 0;
    g.ctl->theta = all ? 0ull : (unsigned long long)th;
  }
}

// Step k of a run from step k0 on: every block reduces step k - 1's per-block results to the pivot p (all blocks reach the
// same p), forms the reflector H = I - tau v v^T from row p's residual x (coordinates k..r-1,
// v = x - alpha e_0, alpha = -sign(x_0) |x|, tau = 1 / (|x|^2 + |x| |x_0|)) in shared memory, and
// reflects its share of the listed rows, recomputing their residual norms (coordinates k+1..).
// Row p itself is left as it is (other blocks read it during this launch): its column of R is
// its coordinates 0..k-1 plus rdiag[k]. Where the list does not hold every unchosen row, the run
// stops (ctl) before a step whose best two listed norms do not both exceed every other row's norm at
// the run's start: a reflection never adds to a row's residual, so until then they are the best two
// of all rows (the margin of 1e-10 is far above the norms' rounding).
//
// A row belongs to W warps, which keep its residual in registers (NREG values per lane) from its
// one read to its one write: dot product, update and norm are three float64 multiply-adds per
// value, at two per clock and SM the bound of this kernel; the rows of Z (67 MB at 4096 x 2048)
// stay in L2. One block per SM; the unchosen rows are kept as a list, dealt to the blocks in turn,
// so that no SM holds more than one row above its share (the chosen row's slot takes the last row).
// 4096 x 4096, r = 2048: the form that this replaced (rows read twice from L2, by warps fixed to
// rows; three more block-wide sums before the first row) took 84.3 us a step against 16 us of
// float64 multiply-adds; this one takes 34 us.
template <int NREG, int W>
constexpr int kGreedyWarps = NREG <= 32 ? 12 : 8;  // what the registers allow
template <int NREG, int W>
__global__ void __launch_bounds__(32 * kGreedyWarps<NREG, W>, 1) greedy_step(Greedy g, int k, int k0) {
  constexpr int WARPS = kGreedyWarps<NREG, W>, GROUPS = WARPS / W, LEN = 32 * NREG * W;
  extern __shared__ double v[];  // LEN entries, zero from r - k on
  __shared__ double part[2][WARPS], s_tau;
  const Top2* in = g.blk + (k & 1) * g.nblk;
  Top2* out = g.blk + ((k + 1) & 1) * g.nblk;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = warp / W, wq = warp % W;
  pdl_launch_dependents();
  pdl_wait_primary();
  if (g.ctl->stop) return;
  const bool all = g.ctl->all;
  const int len = g.r - k, n = g.ctl->count - (k - k0);  // listed rows still unchosen, p among them
  const int c0 = wq * 32 * NREG + lane;
  double y[NREG];
  auto load = [&](int i) {
    const double* z = g.Z + (int64_t)i * g.r + k;
#pragma unroll
    for (int u = 0; u < NREG; ++u) y[u] = c0 + 32 * u < len ? z[c0 + 32 * u] : 0.0;
  };
  const int s0 = blockIdx.x + gridDim.x * grp;
  if (s0 < n - 1) load(g.act[s0]);  // this warp's first row, under the reduction (p's own is replaced)
  Top2 t = top2_empty();
  for (int b = threadIdx.x; b < g.nblk; b += WARPS * 32) top2_merge(t, in[b]);
  t = block_top2(t);
  const int p = t.i1;
  if (!all && (t.i2 < 0 || !(__longlong_as_double((long long)t.v2) >
                             __longlong_as_double((long long)g.ctl->theta) * (1.0 + 1e-10)))) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // every block finds the same, or the flag set
      g.ctl->k_end = k;
      g.ctl->stop = 1;
    }
    return;
  }
  if (p < 0 || p >= g.m || t.s1 < 0 || t.s1 >= n) return;  // cannot happen for m >= r; guards the reads
  const double* zp = g.Z + (int64_t)p * g.r + k;
  const int tail = g.act[n - 1];
  for (int c = threadIdx.x; c < LEN; c += WARPS * 32)
    if (c > 0) v[c] = c < len ? zp[c] : 0.0;
  if (threadIdx.x < 32) {  // one warp: a float64 square root and division by each would delay the rows
    const double nx2 = __longlong_as_double((long long)t.v1), nx = sqrt(nx2);
    const double x0 = zp[0];
    const double alpha = -copysign(nx, x0 != 0.0 ? x0 : 1.0);
    if (threadIdx.x == 0) {
      v[0] = x0 - alpha;
      s_tau = nx2 > 0.0 ? recip(fma(nx, fabs(x0), nx2)) : 0.0;
      if (blockIdx.x == 0 && g.tau) g.tau[k] = s_tau;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      g.order[k] = p;
      g.rdiag[k] = alpha;
      g.sel[p] = 1;          // read only by later launches
      g.act[t.s1] = tail;    // a row loaded early from that slot is loaded again below
    }
  }
  __syncthreads();
  if (blockIdx.x == gridDim.x - 1 && warp == WARPS - 1) {  // the warp with the fewest rows
    const double nx = sqrt(__longlong_as_double((long long)t.v1));
    const double b2 = t.i2 >= 0 ? sqrt(__longlong_as_double((long long)t.v2)) : 0.0;
    if (lane == 0) g.gap[k] = nx > 0.0 ? (nx - b2) / nx : 0.0;
  }
  const double tau = s_tau;
  Top2 mine = top2_empty();
  for (int s = s0; s < n - 1; s += gridDim.x * GROUPS) {
    const int i = s == t.s1 ? tail : g.act[s];
    double* z = g.Z + (int64_t)i * g.r + k;
    if (s != s0 || s == t.s1) load(i);
    double d0 = 0.0, d1 = 0.0;
#pragma unroll
    for (int u = 0; u < NREG; u += 2) {
      d0 = fma(y[u], v[c0 + 32 * u], d0);
      d1 = fma(y[u + 1], v[c0 + 32 * u + 32], d1);
    }
    double d = warp_sum(d0 + d1);
    if (W > 1) {
      if (lane == 0) part[0][warp] = d;
      named_barrier_sync(1 + grp, 32 * W);
      d = 0.0;
#pragma unroll
      for (int w = 0; w < W; ++w) d += part[0][grp * W + w];
    }
    const double f = -tau * d;
    d0 = d1 = 0.0;
#pragma unroll
    for (int u = 0; u < NREG; ++u) {
      y[u] = fma(f, v[c0 + 32 * u], y[u]);
      if (c0 + 32 * u < len) z[c0 + 32 * u] = y[u];
      const double x = u == 0 && c0 == 0 ? 0.0 : y[u];
      if (u & 1) d1 = fma(x, x, d1);
      else d0 = fma(x, x, d0);
    }
    double nr = warp_sum(d0 + d1);
    if (W > 1) {
      if (lane == 0) part[1][warp] = nr;
      named_barrier_sync(1 + grp, 32 * W);
      nr = 0.0;
#pragma unroll
      for (int w = 0; w < W; ++w) nr += part[1][grp * W + w];
    }
    if (lane == 0 && wq == 0) top2_add(mine, norm_key(nr), i, s);
  }
  mine = block_top2(mine);
  if (threadIdx.x == 0) out[blockIdx.x] = mine;
}

// The form of step k for residuals of `len` values: one warp a row up to 2048 values, then 2, 4 or 8
// (2 or 4 warps a row from the start cost 92 / 99 ms of steps against 70 at 4096 x 4096, r = 2048; four
// warps a row for candidate blocks alone gain nothing, 73.3 against 72.6 ms of call).
using GreedyStep = void (*)(Greedy, int, int);
GreedyStep greedy_form(int len, int* threads, size_t* smem) {
  static const GreedyStep one[8] = {greedy_step<8, 1>,  greedy_step<16, 1>, greedy_step<24, 1>, greedy_step<32, 1>,
                                    greedy_step<40, 1>, greedy_step<48, 1>, greedy_step<56, 1>, greedy_step<64, 1>};
  const int u = (len + 255) / 256;  // 8 values per lane each
  *threads = u <= 4 ? 384 : 256;
  if (u <= 8) {
    *smem = (size_t)u * 256 * 8;
    return one[u - 1];
  }
  const int w = u <= 16 ? 2 : u <= 32 ? 4 : 8;
  *smem = (size_t)2048 * w * 8;
  return w == 2 ? greedy_step<64, 2> : w == 4 ? greedy_step<64, 4> : greedy_step<64, 8>;
}

// ---- candidate blocks ----------------------------------------------------------------------------
// A step over every unchosen row costs three float64 multiply-adds per value of Z, but only rows of
// large residual can be chosen, and no residual grows. So, while Z is large, a run of up to kRun steps
// works on the rows of the largest norms alone (greedy_select, greedy_step) and ends when another row
// might come into play; the other rows then take the run's reflectors at once, Z -= W T V^T with
// W = Z V (the compact WY form of Schreiber and Van Loan, 1989; T^-1 = diag(1 / tau) + the strictly upper
// part of V^T V), as two products on the tensor cores and a substitution per row, and all norms are
// recomputed (both products need an error relative to the rows' norms only, as Householder steps have it;
// see run_scale). The pivots, and the order of every comparison that decides one, are those of the
// exhaustive steps. 4096 x 4096, r = 2048: the call 86.1 -> 67.8 ms.
constexpr int kRun = 64;
// Rows of a run: six for every SM. More make a run longer, fewer a step shorter: 65.3 ms of call at
// 4096 x 4096, r = 2048; with 512 rows 69.0, 608 66.2, 760 65.9, 1216 66.2.
constexpr int kCandidates = 912;
constexpr int kRunSlices = 4;  // K-slices of Z V, whose tiles (128 rows each) are few
// Values of Z left (unchosen rows x coordinates) from which on a candidate block pays.
constexpr int64_t kRunFrom = 2000000;

// The power of two by which a run's reflector is scaled, from the pivot's norm |R_kk|: reflectors of norm
// sqrt(2) to 4, whatever the norms of the run's pivots. In Z -= (W T) V^T the slices' errors are relative
// to the largest of a row's weights times the largest of a column's reflector entries; a weight is at most
// tau |v| |z| <= 4 |z|, so that they stay near 2^-58 of |z|, the row's norm, where each step by itself
// rounds to 2^-53 of it. Unscaled, pivots of falling norms in one run (10^6 to 1) made that 2^-38.
__device__ __forceinline__ double run_scale(double rkk) {
  const int ex = (int)(((unsigned long long)__double_as_longlong(rkk) >> 52) & 2047ull);
  return ex < 1 || ex > 2045 ? 1.0 : __longlong_as_double((long long)(2046 - ex) << 52);
}

// V (kRun x len, row-major): row j the scaled reflector of step k0 + j over coordinates k0..r-1, zero rows
// from `steps` on.
__global__ void run_vectors(Greedy g, int k0, int steps, double* V) {
  const int len = g.r - k0, j = blockIdx.y;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= len) return;
  double v = 0.0;
  if (j < steps && c >= j) {
    v = g.Z[(int64_t)g.order[k0 + j] * g.r + k0 + c];
    if (c == j) v -= g.rdiag[k0 + j];
    v *= run_scale(g.rdiag[k0 + j]);
  }
  V[(int64_t)j * len + c] = v;
}

// S[i][j] = v_i . v_j for i < j < kRun, a warp each.
__global__ void __launch_bounds__(256) run_gram(const double* V, int len, double* S) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int i = w / kRun, j = w % kRun;
  if (i >= kRun || i >= j) return;
  const double *a = V + (int64_t)i * len, *b = V + (int64_t)j * len;
  double s0 = 0.0, s1 = 0.0;
  int c = lane;
  for (; c + 32 < len; c += 64) {
    s0 = fma(a[c], b[c], s0);
    s1 = fma(a[c + 32], b[c + 32], s1);
  }
  if (c < len) s0 = fma(a[c], b[c], s0);
  s0 = warp_sum(s0 + s1);
  if (lane == 0) S[i * kRun + j] = s0;
}

// W (m x kRun, the sum of its slices) becomes W T by forward substitution, w_j = tau_j (w_j - sum over i < j of w_i S[i][j]),
// and zero for the rows that already carry the run's reflectors (listed) or must not (chosen before).
// Four lanes a row, each with every fourth column.
__global__ void __launch_bounds__(128) run_substitute(Greedy g, int k0, int steps, const double* S, const uint8_t* in_list,
                                                      double* W, int slices) {
  __shared__ double s_S[kRun * kRun];
  __shared__ double s_tau[kRun];
  for (int e = threadIdx.x; e < kRun * kRun; e += 128) s_S[e] = e / kRun < e % kRun ? S[e] : 0.0;
  if (threadIdx.x < kRun) {
    double t = 0.0;
    if ((int)threadIdx.x < steps) {
      const double back = 1.0 / run_scale(g.rdiag[k0 + threadIdx.x]);  // V's reflector is scaled
      t = g.tau[k0 + threadIdx.x] * back * back;
    }
    s_tau[threadIdx.x] = t;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int row = blockIdx.x * 32 + (threadIdx.x >> 2);
  const bool live = row < g.m && !g.sel[row] && !in_list[row];
  double w[kRun / 4];
  double* p = W + (int64_t)row * kRun;
#pragma unroll
  for (int u = 0; u < kRun / 4; ++u) w[u] = live ? p[4 * u + q] : 0.0;
  for (int z = 1; z < slices; ++z)  // Z V came in K-slices
#pragma unroll
    for (int u = 0; u < kRun / 4; ++u)
      if (live) w[u] += p[(int64_t)z * g.m * kRun + 4 * u + q];
#pragma unroll
  for (int j = 0; j < kRun; ++j) {
    const double x = __shfl_sync(0xffffffffu, w[j / 4], (lane & ~3) | (j & 3)) * s_tau[j];
    if (q == (j & 3)) w[j / 4] = x;
#pragma unroll
    for (int u = j / 4; u < kRun / 4; ++u)
      if (4 * u + q > j) w[u] = fma(-x, s_S[j * kRun + 4 * u + q], w[u]);
  }
  if (row < g.m)
#pragma unroll
    for (int u = 0; u < kRun / 4; ++u) p[4 * u + q] = w[u];
}

// Doubles of scratch a candidate block needs beside the sliced operands: V, S, W, tau; and, for every
// form, the rows' norms and flags.
int64_t run_doubles(int64_t m, int64_t r) { return kRun * r + kRun * kRun + kRunSlices * kRun * m + r + 64; }

// ---- R, its inverse, the index sets -----------------------------------------------------------
// R (rp x rp, row-major, upper triangular, selection order): R[c][k] = Z[order[k]][c] for c < k,
// R[k][k] = rdiag[k]; identity on the padding k >= r.
__global__ void build_r(const Greedy g, double* R, int rp) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)rp * rp) return;
  const int c = (int)(e / rp), k = (int)(e % rp);
  double val = 0.0;
  if (k >= g.r) {
    val = c == k ? 1.0 : 0.0;
  } else if (c < k) {
    val = g.Z[(int64_t)g.order[k] * g.r + c];
  } else if (c == k) {
    val = g.rdiag[k];
  }
  R[e] = val;
}

// Inverses of the 32 x 32 diagonal blocks of R into Rinv (whose other entries are zeroed): thread
// j of block b solves R_bb y = e_j by back substitution.
__global__ void inv_diag32(const double* R, double* Rinv, int rp) {
  __shared__ double Rb[32][33];
  __shared__ double Y[32][33];
  const int b = blockIdx.x, j = threadIdx.x;
  const int64_t base = (int64_t)b * 32;
  for (int i = 0; i < 32; ++i) Rb[i][j] = R[(base + i) * rp + base + j];
  __syncthreads();
  for (int i = 31; i >= 0; --i) {
    double s = (i == j) ? 1.0 : 0.0;
    for (int l = i + 1; l <= j; ++l) s -= Rb[i][l] * Y[l][j];
    Y[i][j] = i <= j ? s / Rb[i][i] : 0.0;
  }
  __syncthreads();
  for (int i = 0; i < 32; ++i) Rinv[(base + i) * rp + base + j] = Y[i][j];
}

// Ascending I and I^c from the chosen-row flags, and for every selection step k the position of
// its row in ascending I (one block of 1024 threads, chunked prefix sums).
__global__ void __launch_bounds__(1024) index_sets(const int32_t* sel, int m, const int32_t* order, int r,
                                                   int32_t* piv, int32_t* nonpiv, int32_t* pos, int32_t* asc) {
  __shared__ int s_cnt[1024];
  __shared__ int s_base;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  for (int c0 = 0; c0 < m; c0 += 1024) {
    const int i = c0 + threadIdx.x;
    const int f = (i < m && sel[i]) ? 1 : 0;
    s_cnt[threadIdx.x] = f;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {  // inclusive scan
      const int v = threadIdx.x >= o ? s_cnt[threadIdx.x - o] : 0;
      __syncthreads();
      s_cnt[threadIdx.x] += v;
      __syncthreads();
    }
    if (i < m) {
      const int before = s_base + s_cnt[threadIdx.x] - f;  // chosen rows before i
      pos[i] = before;
      if (f) {
        if (before < r) piv[before] = i;
      } else if (i - before < m - r) {
        nonpiv[i - before] = i;
      }
    }
    __syncthreads();
    if (threadIdx.x == 1023) s_base += s_cnt[1023];
    __syncthreads();
  }
  for (int k = threadIdx.x; k < r; k += 1024) asc[k] = pos[order[k]];
}

// max |C| over the (m - r) x r block (non-negative doubles order like their bit patterns).
__global__ void max_abs(const double* C, int64_t rows, int64_t cols, int64_t ldc, unsigned long long* out) {
  double mx = 0.0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += (int64_t)gridDim.x * blockDim.x)
    mx = fmax(mx, fabs(C[(e / cols) * ldc + e % cols]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(mx));
}

// Rinv = R^{-1} for an upper-triangular R (rp x rp, rp = 32 * 2^k; identity on any padding), by
// doubling: the 32 x 32 diagonal blocks inverted directly, then, level by level, for every pair
// of sz-blocks [[A, B], [0, D]] along the diagonal the off-diagonal block -A^{-1} (B D^{-1}).
// Tt: scratch of rp * rp / 4 doubles; `scratch` for the sliced operands of the levels from 512 on
// (below, all pairs of a level go in one batched launch on the CUDA cores: 256-blocks, r = 2048, eight
// products 260 us in two launches, one by one in slices 376).
int upper_inverse(const double* R, double* Rinv, double* Tt, int rp, void* scratch, int64_t bytes, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(Rinv, 0, (size_t)rp * rp * 8, s);
  if (e != cudaSuccess) return pifa_fail_cuda("upper inverse: memset", e);
  inv_diag32<<<rp / 32, 32, 0, s>>>(R, Rinv, rp);
  pifa_count_launch();
  e = cudaGetLastError();
  if (e != cudaSuccess) return pifa_fail_cuda("upper inverse: launch", e);
  int st;
  for (int sz = 32; sz < rp; sz *= 2) {
    const int pairs = rp / (2 * sz);
    const int64_t step = (int64_t)2 * sz * rp + 2 * sz;  // next pair along the diagonal
    GemmF64 a = {};
    a.M = sz; a.N = sz; a.K = sz;
    a.A = R + sz; a.sa_i = rp; a.sa_k = 1;                        // B block
    a.B = Rinv + (int64_t)sz * rp + sz; a.sb_k = rp; a.sb_j = 1;  // D^{-1}
    a.C = Tt; a.ldc = sz; a.alpha = 1.0; a.beta = 0.0; a.tri = 2;
    a.za = step; a.zb = step; a.zc = (int64_t)sz * sz;
    GemmF64 b = {};
    b.M = sz; b.N = sz; b.K = sz;
    b.A = Rinv; b.sa_i = rp; b.sa_k = 1;                          // A^{-1}
    b.B = Tt; b.sb_k = sz; b.sb_j = 1;
    b.C = Rinv + sz; b.ldc = rp; b.alpha = -1.0; b.beta = 0.0; b.tri = 4;
    b.za = step; b.zb = (int64_t)sz * sz; b.zc = step;
    if (sz < 512 || !gemm_f64_split_fits(a, bytes) || !gemm_f64_split_fits(b, bytes)) {
      if ((st = run_gemm_f64(a, pairs, s)) != PIFA_OK || (st = run_gemm_f64(b, pairs, s)) != PIFA_OK) return st;
      continue;
    }
    for (int z = 0; z < pairs; ++z) {
      if ((st = gemm_f64_split(a, scratch, bytes, s)) != PIFA_OK || (st = gemm_f64_split(b, scratch, bytes, s)) != PIFA_OK)
        return st;
      a.A += a.za; a.B += a.zb; a.C += a.zc;
      b.A += b.za; b.B += b.zb; b.C += b.zc;
    }
  }
  return PIFA_OK;
}

// Workspace layout (bytes, each part 256-aligned).
struct Layout {
  int64_t G, L, Z, R, Rinv, T, blk, order, rdiag, gap, sel, pos, asc, flags, total;
  int rp, nblk;
};

int64_t a256(int64_t b) { return (b + 255) / 256 * 256; }

Layout layout(int64_t m, int64_t r) {
  Layout L = {};
  int rp = 32;
  while (rp < r) rp *= 2;
  L.rp = rp;
  L.nblk = 4 * 152;
  int64_t o = 0;
  auto take = [&](int64_t bytes) {
    const int64_t at = o;
    o += a256(bytes);
    return at;
  };
  L.G = take(r * r * 8);
  L.L = take(r * r * 8);
  L.Z = take(m * r * 8);
  L.R = take((int64_t)rp * rp * 8);
  L.Rinv = take((int64_t)rp * rp * 8);
  L.T = take((int64_t)rp * rp / 4 * 8 + 8);
  L.blk = take(2 * (int64_t)L.nblk * (int64_t)sizeof(Top2));
  L.order = take(r * 4);
  L.rdiag = take(r * 8);
  L.gap = take(r * 8);
  L.sel = take(m * 4);
  L.pos = take(m * 4);
  L.asc = take(r * 4);
  L.flags = take(64);
  L.total = o;
  return L;
}

constexpr int64_t kMaxRank = 16384;  // the reflector lives in shared memory (r doubles)

}  // namespace

int gemm_f64_flagged(const GemmF64& p, const uint32_t* mask, int words, cudaStream_t s) {
  gemm_f64_masked<<<dim3((unsigned)((p.N + 31) / 32), (unsigned)((p.M + 31) / 32)), 256, 0, s>>>(p, mask, words);
  pifa_count_launch();
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PIFA_OK : pifa_fail_cuda("float64 products: flagged elements", e);
}

extern "C" int64_t pifa_compress_device_workspace_size(int64_t m, int64_t n, int64_t r) {
  pifa_clear_error();
  if (m < 1 || n < 1 || r < 1 || r > m || r > n) return pifa_fail(PIFA_ERR_INVALID_ARG, "need 1 <= r <= min(m, n)");
  if (r > kMaxRank || m >= ((int64_t)1 << 30) || n >= ((int64_t)1 << 30))
    return pifa_fail(PIFA_ERR_UNSUPPORTED, "pifa_compress_device needs r <= 16384 and m, n < 2^30");
  return layout(m, r).total;
}

extern "C" int pifa_compress_device(const double* U, const double* V, int64_t m, int64_t n, int64_t r,
                                    int32_t* pivot_idx, int32_t* nonpivot_idx, double* Wp, int64_t ldwp,
                                    double* C, int64_t ldc, void* workspace, int64_t workspace_bytes,
                                    pifa_compress_info* info, void* cuda_stream) {
  const int64_t need = pifa_compress_device_workspace_size(m, n, r);
  if (need < 0) return (int)need;
  pifa_clear_error();
  const bool has_np = m > r;
  if (!U || !V || !pivot_idx || !Wp || (has_np && (!nonpivot_idx || !C)))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "null U, V, pivot_idx, Wp, nonpivot_idx or C");
  if (ldwp < n || (has_np && ldc < r)) return pifa_fail(PIFA_ERR_INVALID_ARG, "leading dimension smaller than the row");
  if (!workspace || workspace_bytes < need) return pifa_fail(PIFA_ERR_WORKSPACE, "workspace missing or too small");
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return pifa_fail(PIFA_ERR_ALIGNMENT, "workspace must be 256-byte aligned");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  const Layout Ly = layout(m, r);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  double* G = reinterpret_cast<double*>(ws + Ly.G);
  double* L = reinterpret_cast<double*>(ws + Ly.L);
  double* Z = reinterpret_cast<double*>(ws + Ly.Z);
  double* R = reinterpret_cast<double*>(ws + Ly.R);
  double* Rinv = reinterpret_cast<double*>(ws + Ly.Rinv);
  double* Tt = reinterpret_cast<double*>(ws + Ly.T);
  int* flags = reinterpret_cast<int*>(ws + Ly.flags);  // [0] Cholesky failure, [2..3] max |C| bits
  Greedy g;
  g.Z = Z;
  g.m = (int)m;
  g.r = (int)r;
  g.sel = reinterpret_cast<int32_t*>(ws + Ly.sel);
  g.act = reinterpret_cast<int32_t*>(ws + Ly.pos);  // index_sets fills it afresh afterwards
  g.blk = reinterpret_cast<Top2*>(ws + Ly.blk);
  g.nblk = kGreedyBlocks;
  g.order = reinterpret_cast<int32_t*>(ws + Ly.order);
  g.rdiag = reinterpret_cast<double*>(ws + Ly.rdiag);
  g.gap = reinterpret_cast<double*>(ws + Ly.gap);
  int32_t* pos = reinterpret_cast<int32_t*>(ws + Ly.pos);
  int32_t* asc = reinterpret_cast<int32_t*>(ws + Ly.asc);
  const int ri = (int)r, mi = (int)m, ni = (int)n, rp = Ly.rp;
  cudaError_t e;
  int st;
#define PIFA_CK(call, what)                          \
  do {                                               \
    if ((e = (call)) != cudaSuccess) return pifa_fail_cuda(what, e); \
  } while (0)
  PIFA_CK(cudaMemsetAsync(flags, 0, 64, s), "compress: memset");
  PIFA_CK(cudaMemsetAsync(g.sel, 0, m * 4, s), "compress: memset");
  PIFA_CK(cudaMemsetAsync(L, 0, r * r * 8, s), "compress: memset");
  // every index a later kernel gathers through starts valid, whatever the selection does
  PIFA_CK(cudaMemsetAsync(g.order, 0, r * 4, s), "compress: memset");
  PIFA_CK(cudaMemsetAsync(pivot_idx, 0, r * 4, s), "compress: memset");
  if (has_np) PIFA_CK(cudaMemsetAsync(nonpivot_idx, 0, (m - r) * 4, s), "compress: memset");

  // 1. G = V^T V, L = chol(G), Z = U L
  GemmF64 q = {};
  q.M = ri; q.N = ri; q.K = ni;
  q.A = V; q.sa_i = 1; q.sa_k = r;
  q.B = V; q.sb_k = r; q.sb_j = 1;
  q.C = G; q.ldc = r; q.alpha = 1.0; q.beta = 0.0;
  q.lower = 1;  // G is symmetric
  // scratch of the products: parts of the workspace that hold nothing yet, or nothing any more
  if ((st = run_product(q, Z, Ly.blk - Ly.Z, s)) != PIFA_OK) return st;
  if ((st = cholesky(G, L, r, flags, Z, Ly.blk - Ly.Z, s)) != PIFA_OK) return st;
  q = GemmF64{};
  q.M = mi; q.N = ri; q.K = ri;
  q.A = U; q.sa_i = r; q.sa_k = 1;
  q.B = L; q.sb_k = r; q.sb_j = 1;
  q.C = Z; q.ldc = r; q.alpha = 1.0; q.beta = 0.0; q.tri = 1;
  if ((st = run_product(q, R, Ly.blk - Ly.R, s)) != PIFA_OK) return st;

  // 2. r greedy steps
  g.ctl = reinterpret_cast<GreedyCtl*>(flags + 4);
  auto run_steps = [&](int from, int to) {
    for (int j = from; j < to; ++j) {
      cudaLaunchConfig_t cfg = {};
      int threads = 0;
      const GreedyStep step = greedy_form(ri - j, &threads, &cfg.dynamicSmemBytes);
      if (cfg.dynamicSmemBytes > 32768 &&
          (e = cudaFuncSetAttribute(step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes)) != cudaSuccess)
        return pifa_fail_cuda("compress: greedy smem attribute", e);
      cfg.gridDim = dim3((unsigned)g.nblk);
      cfg.blockDim = dim3((unsigned)threads);
      cfg.stream = s;
      cudaLaunchAttribute attr;  // the next step's launch overlaps this step's tail
      attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr.val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      if ((e = pifa_launch_ex(&cfg, step, g, j, from)) != cudaSuccess)
        return pifa_fail_cuda("compress: greedy step launch", e);
    }
    return (int)PIFA_OK;
  };
  // Candidate blocks: the norms and flags where R goes later, the sliced operands behind them, the
  // small matrices where G and L were.
  double* norms = R;
  uint8_t* in_list = reinterpret_cast<uint8_t*>(norms + m);
  uint8_t* slices = ws + Ly.R + a256(m * 9);
  const int64_t slice_bytes = Ly.blk - Ly.R - a256(m * 9);
  double *V_run = G, *S_run = V_run + kRun * r, *W_run = S_run + kRun * kRun, *tau_run = W_run + kRunSlices * kRun * m;
  const bool runs = r >= 256 && slice_bytes > 0 && run_doubles(m, r) * 8 <= Ly.Z - Ly.G && m * r >= kRunFrom;
  int k = 0, guess = kRun;
  for (bool more = runs; more;) {
    const bool block = (int64_t)(mi - k) * (ri - k) >= kRunFrom;  // else: every row, to the end
    const int most = guess < kRun ? guess : kRun;  // a run's length changes slowly: few launches find it over
    const int steps = block && ri - k > most ? most : ri - k;
    g.tau = block ? tau_run : nullptr;
    greedy_norms<<<4 * kGreedyBlocks, 256, 0, s>>>(g, k, norms);
    pifa_count_launch();
    greedy_select<<<1, 1024, 0, s>>>(g, k, norms, block ? kCandidates : 0, block ? in_list : nullptr);
    pifa_count_launch();
    PIFA_CK(cudaGetLastError(), "compress: greedy selection launch");
    if ((st = run_steps(k, k + steps)) != PIFA_OK) return st;
    if (!block) {
      k = ri;
      break;
    }
    GreedyCtl c = {};
    PIFA_CK(cudaMemcpyAsync(&c, g.ctl, sizeof c, cudaMemcpyDeviceToHost, s), "compress: read back");
    PIFA_CK(cudaStreamSynchronize(s), "compress: synchronize");
    const int done = c.stop ? c.k_end - k : steps;
    if (done <= 0 || done > steps) break;  // no step was sure: the rest exhaustively
    if (!c.all) {  // the other rows take the run's reflectors
      const int len = ri - k;
      run_vectors<<<dim3((unsigned)((len + 255) / 256), kRun), 256, 0, s>>>(g, k, done, V_run);
      pifa_count_launch();
      run_gram<<<kRun * kRun / 8, 256, 0, s>>>(V_run, len, S_run);
      pifa_count_launch();
      GemmF64 w = {};  // W = Z V
      w.M = mi; w.N = kRun; w.K = len;
      w.A = Z + k; w.sa_i = r; w.sa_k = 1;
      w.B = V_run; w.sb_k = 1; w.sb_j = len;
      w.C = W_run; w.ldc = kRun; w.alpha = 1.0; w.beta = 0.0; w.normwise = 1;
      const int parts = gemm_f64_split_fits(w, slice_bytes) ? kRunSlices : 1;
      st = parts > 1 ? gemm_f64_split(w, slices, slice_bytes, s, parts, m * kRun) : run_gemm_f64(w, 1, s);
      if (st != PIFA_OK) return st;
      run_substitute<<<(unsigned)((m + 31) / 32), 128, 0, s>>>(g, k, done, S_run, in_list, W_run, parts);
      pifa_count_launch();
      GemmF64 u = {};  // Z -= (W T) V^T
      u.M = mi; u.N = len; u.K = kRun;
      u.A = W_run; u.sa_i = kRun; u.sa_k = 1;
      u.B = V_run; u.sb_k = len; u.sb_j = 1;
      u.C = Z + k; u.ldc = r; u.alpha = -1.0; u.beta = 1.0; u.normwise = 1;
      if ((st = run_product(u, slices, slice_bytes, s)) != PIFA_OK) return st;
      PIFA_CK(cudaGetLastError(), "compress: candidate block launch");
    }
    k += done;
    guess = done + 8;
    more = k < ri;
  }
  if (k < ri) {  // every step over every row
    g.tau = nullptr;
    if (k == 0) {
      greedy_init<<<g.nblk, 256, 0, s>>>(g);
    } else {
      greedy_norms<<<4 * kGreedyBlocks, 256, 0, s>>>(g, k, norms);
      pifa_count_launch();
      greedy_select<<<1, 1024, 0, s>>>(g, k, norms, 0, nullptr);
    }
    pifa_count_launch();
    PIFA_CK(cudaGetLastError(), "compress: greedy init launch");
    if ((st = run_steps(k, ri)) != PIFA_OK) return st;
  }

  // 3. index sets, R, R^{-1}, C = Z[I^c] R^{-T} in ascending-I columns
  index_sets<<<1, 1024, 0, s>>>(g.sel, mi, g.order, ri, pivot_idx, has_np ? nonpivot_idx : pos, pos, asc);
  pifa_count_launch();
  PIFA_CK(cudaGetLastError(), "compress: index sets launch");
  {
    const int64_t tot = (int64_t)rp * rp;
    build_r<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(g, R, rp);
    pifa_count_launch();
    if ((st = upper_inverse(R, Rinv, Tt, rp, G, Ly.Z - Ly.G, s)) != PIFA_OK) return st;  // G and L are done with
  }
  if (has_np) {
    // C[a][asc[j]] = sum_{k >= j} Z[I^c[a]][k] Rinv[j][k]
    GemmF64 c = {};
    c.M = (int)(m - r); c.N = ri; c.K = ri;
    c.A = Z; c.aidx = nonpivot_idx; c.sa_i = r; c.sa_k = 1;
    c.B = Rinv; c.sb_k = 1; c.sb_j = rp;
    c.C = C; c.cidx = asc; c.ldc = ldc; c.alpha = 1.0; c.beta = 0.0; c.tri = 1;
    if ((st = run_product(c, G, Ly.Z - Ly.G, s)) != PIFA_OK) return st;
    max_abs<<<4 * 152, 256, 0, s>>>(C, m - r, r, ldc, reinterpret_cast<unsigned long long*>(flags + 2));
    pifa_count_launch();
    PIFA_CK(cudaGetLastError(), "compress: max launch");
  }
  // 4. W_p = U[I] V^T
  {
    GemmF64 w = {};
    w.M = ri; w.N = ni; w.K = ri;
    w.A = U; w.aidx = pivot_idx; w.sa_i = r; w.sa_k = 1;
    w.B = V; w.sb_k = 1; w.sb_j = r;
    w.C = Wp; w.ldc = ldwp; w.alpha = 1.0; w.beta = 0.0;
    if ((st = run_product(w, G, Ly.blk - Ly.G, s)) != PIFA_OK) return st;
  }

  // results for the rank check and the diagnostics
  int hflags[4] = {0, 0, 0, 0};
  double rd0 = 0.0, rdl = 0.0;
  PIFA_CK(cudaMemcpyAsync(hflags, flags, sizeof hflags, cudaMemcpyDeviceToHost, s), "compress: read back");
  PIFA_CK(cudaMemcpyAsync(&rd0, g.rdiag, 8, cudaMemcpyDeviceToHost, s), "compress: read back");
  PIFA_CK(cudaMemcpyAsync(&rdl, g.rdiag + (r - 1), 8, cudaMemcpyDeviceToHost, s), "compress: read back");
  double* hgap = nullptr;
  PIFA_CK(cudaMallocHost(&hgap, r * 8), "compress: host buffer");
  e = cudaMemcpyAsync(hgap, g.gap, r * 8, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  double min_gap = 1.0;
  if (e == cudaSuccess)
    for (int64_t k = 0; k < r; ++k) min_gap = hgap[k] < min_gap ? hgap[k] : min_gap;
  cudaFreeHost(hgap);
  if (e != cudaSuccess) return pifa_fail_cuda("compress: synchronize", e);
#undef PIFA_CK
  double cmax = 0.0;
  {
    unsigned long long bits = (unsigned long long)(unsigned)hflags[2] | ((unsigned long long)(unsigned)hflags[3] << 32);
    memcpy(&cmax, &bits, 8);
  }
  if (info) {
    info->min_pivot_gap = min_gap;
    info->r_ratio = rd0 != 0.0 ? std::fabs(rdl) / std::fabs(rd0) : 0.0;
    info->max_abs_c = cmax;
    info->threads = 0;
  }
  if (hflags[0] || !(std::fabs(rdl) >= 1e-8 * std::fabs(rd0)) || rd0 == 0.0)
    return pifa_fail(PIFA_ERR_RANK_DEFICIENT, "W' = U V^T has fewer than r independent rows (|R_rr| < 1e-8 |R_00|)");
  return PIFA_OK;
}

// ---- the M reconstruction solves (Sec. 4, Eqs. 4 and 8; Algorithm 3, part 1) ------------------
namespace {

// dst (rows x cols, pitch lddst, fp64) = src (fp32, pitch ldsrc)
__global__ void f32_to_f64(const float* src, int64_t ldsrc, int64_t rows, int64_t cols, double* dst, int64_t lddst) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += (int64_t)gridDim.x * blockDim.x)
    dst[(e / cols) * lddst + e % cols] = (double)src[(e / cols) * ldsrc + e % cols];
}

// dst (rows x cols, fp64) += alpha * W (bf16, pitch ldw)
__global__ void add_scaled_bf16(const __nv_bfloat16* W, int64_t ldw, int64_t rows, int64_t cols, double alpha,
                                double* dst, int64_t lddst) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += (int64_t)gridDim.x * blockDim.x)
    dst[(e / cols) * lddst + e % cols] += alpha * (double)__bfloat162float(W[(e / cols) * ldw + e % cols]);
}

// A[i][j] = A[j][i] for i > j (n x n, pitch lda): the lower triangle from the upper.
__global__ void mirror_upper(double* A, int64_t n, int64_t lda) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, j = e % n;
    if (i > j) A[i * lda + j] = A[j * lda + i];
  }
}

__global__ void add_diag(double* A, int64_t k, int64_t lda, double alpha) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x)
    A[i * lda + i] += alpha;
}

// R (rp x rp) = L^T for a lower-triangular L (k x k, pitch k), identity on the padding i >= k.
__global__ void transpose_pad_lower(const double* L, int64_t k, double* R, int rp) {
  const int64_t tot = (int64_t)rp * rp;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / rp, j = e % rp;
    double v = 0.0;
    if (i < k && j < k)
      v = i <= j ? L[j * k + i] : 0.0;
    else if (i == j)
      v = 1.0;
    R[e] = v;
  }
}

int grid_for(int64_t work) {
  const int64_t b = (work + 255) / 256;
  return (int)(b < 4 * 152 ? (b > 0 ? b : 1) : 4 * 152);
}

int pad_pow2_32(int64_t k) {
  int rp = 32;
  while (rp < k) rp *= 2;
  return rp;
}

// Scratch of spd_inverse for k: a copy of S, L, R and R^{-1} (rp x rp), and the doubling's T.
int64_t spd_scratch_doubles(int64_t k) {
  const int64_t rp = pad_pow2_32(k);
  return 2 * k * k + 2 * rp * rp + rp * rp / 4 + 64;
}

// Sinv = S^{-1} for a symmetric positive definite S (k x k, pitch k): S = L L^T, R = L^T, S^{-1} = R^{-1} R^{-T}. `bad` is set when a pivot is not positive.
int spd_inverse(const double* S, int64_t k, double* Sinv, double* scratch, int* bad, cudaStream_t s) {
  const int rp = pad_pow2_32(k);
  double* G = scratch;
  double* L = G + k * k;
  double* R = L + k * k;
  double* Rinv = R + (int64_t)rp * rp;
  double* Tt = Rinv + (int64_t)rp * rp;
  cudaError_t e = cudaMemcpyAsync(G, S, (size_t)k * k * 8, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(L, 0, (size_t)k * k * 8, s);
  if (e != cudaSuccess) return pifa_fail_cuda("spd inverse: copy", e);
  const int64_t gl = 2 * k * k * 8, rt = (2 * (int64_t)rp * rp + (int64_t)rp * rp / 4) * 8;  // bytes of G, L and of R .. Tt
  int st = cholesky(G, L, k, bad, R, rt, s);
  if (st != PIFA_OK) return st;
  transpose_pad_lower<<<grid_for((int64_t)rp * rp), 256, 0, s>>>(L, k, R, rp);
  pifa_count_launch();
  e = cudaGetLastError();
  if (e != cudaSuccess) return pifa_fail_cuda("spd inverse: launch", e);
  if ((st = upper_inverse(R, Rinv, Tt, rp, G, gl, s)) != PIFA_OK) return st;  // G and L are done with
  GemmF64 g = {};  // Sinv[i][j] = sum over t >= max(i, j) of Rinv[i][t] Rinv[j][t]
  g.M = (int)k; g.N = (int)k; g.K = (int)k;
  g.A = Rinv; g.sa_i = rp; g.sa_k = 1;
  g.B = Rinv; g.sb_k = 1; g.sb_j = rp;
  g.C = Sinv; g.ldc = k; g.alpha = 1.0; g.beta = 0.0; g.tri = 1 | 4;
  return run_product(g, G, gl, s);
}

}  // namespace

extern "C" int64_t pifa_m_reconstruct_workspace_size(int64_t m, int64_t n, int64_t r) {
  pifa_clear_error();
  if (m < 1 || n < 1 || r < 1 || r > n || r > m) return pifa_fail(PIFA_ERR_INVALID_ARG, "need 1 <= r <= min(m, n)");
  if (n > 16384 || m >= ((int64_t)1 << 30)) return pifa_fail(PIFA_ERR_UNSUPPORTED, "pifa_m_reconstruct needs n <= 16384");
  const int64_t d = 2 * n * n + m * n + n * r + m * r + 4 * r * r + 2 * r * n + spd_scratch_doubles(n > r ? n : r) + 64;
  return d * 8 + 256;
}

extern "C" int pifa_m_reconstruct(const float* XXt, int64_t ldxx, const float* YtXt, int64_t ldyx, const double* V,
                                  const void* W, int64_t ldw, int64_t m, int64_t n, int64_t r, double alpha,
                                  double* U_r, double* V_r, void* workspace, int64_t workspace_bytes,
                                  void* cuda_stream) {
  const int64_t need = pifa_m_reconstruct_workspace_size(m, n, r);
  if (need < 0) return (int)need;
  pifa_clear_error();
  if (!XXt || !YtXt || !V || !U_r || !V_r || (alpha != 0.0 && !W))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "null XXt, YtXt, V, U_r, V_r, or W with alpha != 0");
  if (!(alpha >= 0.0)) return pifa_fail(PIFA_ERR_INVALID_ARG, "alpha must be >= 0");
  if (ldxx < n || ldyx < n || (W && ldw < n)) return pifa_fail(PIFA_ERR_INVALID_ARG, "leading dimension smaller than the row");
  if (!workspace || workspace_bytes < need) return pifa_fail(PIFA_ERR_WORKSPACE, "workspace missing or too small");
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return pifa_fail(PIFA_ERR_ALIGNMENT, "workspace must be 256-byte aligned");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  double* A = static_cast<double*>(workspace);  // X X^T (n x n), later X X^T + alpha I
  double* B = A + n * n;                         // Y_t X^T (m x n), later + alpha W
  double* T1 = B + m * n;                        // X X^T V (n x r)
  double* Sm = T1 + n * r;                       // V^T X X^T V (r x r)
  double* B1 = Sm + r * r;                       // Y_t X^T V (m x r)
  double* Sinv = B1 + m * r;
  double* Pm = Sinv + r * r;                     // U_r^T U_r
  double* Pinv = Pm + r * r;
  double* Rhs = Pinv + r * r;                    // U_r^T (Y_t X^T + alpha W) (r x n)
  double* Q = Rhs + r * n;                       // (U_r^T U_r)^{-1} Rhs (r x n)
  double* Ginv = Q + r * n;                      // (X X^T + alpha I)^{-1}
  int* bad = reinterpret_cast<int*>(Ginv + n * n);
  double* scratch = reinterpret_cast<double*>(bad) + 8;
  cudaError_t e = cudaMemsetAsync(bad, 0, 8, s);
  if (e != cudaSuccess) return pifa_fail_cuda("reconstruct: memset", e);
  f32_to_f64<<<grid_for(n * n), 256, 0, s>>>(XXt, ldxx, n, n, A, n);
  pifa_count_launch();
  mirror_upper<<<grid_for(n * n), 256, 0, s>>>(A, n, n);  // pifa_m_accumulate keeps the upper triangle
  pifa_count_launch();
  f32_to_f64<<<grid_for(m * n), 256, 0, s>>>(YtXt, ldyx, m, n, B, n);
  pifa_count_launch();
  e = cudaGetLastError();
  if (e != cudaSuccess) return pifa_fail_cuda("reconstruct: launch", e);
  const int ni = (int)n, mi = (int)m, ri = (int)r;
  const int64_t sbytes = spd_scratch_doubles(n) * 8;
  int st;
  auto gemm = [&](int M, int N, int K, const double* Ap, int64_t sai, int64_t sak, const double* Bp, int64_t sbk,
                  int64_t sbj, double* Cp, int64_t ldc) {
    GemmF64 g = {};
    g.M = M; g.N = N; g.K = K;
    g.A = Ap; g.sa_i = sai; g.sa_k = sak;
    g.B = Bp; g.sb_k = sbk; g.sb_j = sbj;
    g.C = Cp; g.ldc = ldc; g.alpha = 1.0; g.beta = 0.0;
    return run_product(g, scratch, sbytes, s);  // between the inverses their scratch is free
  };
  // Eq. 4: U_r = (Y_t X^T) V (V^T (X X^T) V)^{-1}
  if ((st = gemm(ni, ri, ni, A, n, 1, V, r, 1, T1, r)) != PIFA_OK) return st;
  if ((st = gemm(ri, ri, ni, V, 1, r, T1, r, 1, Sm, r)) != PIFA_OK) return st;   // V^T T1
  if ((st = gemm(mi, ri, ni, B, n, 1, V, r, 1, B1, r)) != PIFA_OK) return st;
  if ((st = spd_inverse(Sm, r, Sinv, scratch, bad, s)) != PIFA_OK) return st;
  if ((st = gemm(mi, ri, ri, B1, r, 1, Sinv, r, 1, U_r, r)) != PIFA_OK) return st;
  // Eq. 8: V_r^T = (U_r^T U_r)^{-1} U_r^T (Y_t X^T + alpha W) (X X^T + alpha I)^{-1}
  if ((st = gemm(ri, ri, mi, U_r, 1, r, U_r, r, 1, Pm, r)) != PIFA_OK) return st;   // U_r^T U_r
  if ((st = spd_inverse(Pm, r, Pinv, scratch, bad, s)) != PIFA_OK) return st;
  if (alpha != 0.0) {
    add_scaled_bf16<<<grid_for(m * n), 256, 0, s>>>(static_cast<const __nv_bfloat16*>(W), ldw, m, n, alpha, B, n);
    pifa_count_launch();
    add_diag<<<grid_for(n), 256, 0, s>>>(A, n, n, alpha);
    pifa_count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return pifa_fail_cuda("reconstruct: launch", e);
  }
  if ((st = gemm(ri, ni, mi, U_r, 1, r, B, n, 1, Rhs, n)) != PIFA_OK) return st;   // U_r^T B
  if ((st = gemm(ri, ni, ri, Pinv, r, 1, Rhs, n, 1, Q, n)) != PIFA_OK) return st;
  if ((st = spd_inverse(A, n, Ginv, scratch, bad, s)) != PIFA_OK) return st;
  // V_r = (Q Ginv)^T = Ginv Q^T (Ginv symmetric)
  if ((st = gemm(ni, ri, ni, Ginv, n, 1, Q, 1, n, V_r, r)) != PIFA_OK) return st;
  int hbad = 0;
  e = cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return pifa_fail_cuda("reconstruct: synchronize", e);
  if (hbad) return pifa_fail(PIFA_ERR_RANK_DEFICIENT, "a matrix of the reconstruction is not positive definite");
  return PIFA_OK;
}
