// backward.cu -- the gradients of a PIFA layer (fine-tuning after compression, Sec. 5.1; the layer
// is differentiable, Sec. 6) and the online accumulators of the M reconstruction (Sec. 4; the
// accumulation steps of Algorithm 3), as tensor-core contractions (gemm_tc.cu) plus a column split.
//
// Backward, tokens as rows (Y = X W'^T, Y_p = X W_p^T, Y_np = Y_p C^T), given dY = dL/dY:
//   dY_I = dY[:, I], dY_np = dY[:, I^c]      one pass over dY       (Algorithm 2, steps 4-5, reversed)
//   dY_p  = dY_I + dY_np C                   T x r,  K = m - r      (steps 4 and 3, reversed)
//   dX    = dY_p W_p                         T x n,  K = r          (step 2, reversed)
// dY_p and Y_p are kept as hi + lo pairs of bf16 planes: in exact arithmetic dX = dY W', and the
// route through dY_p (amplified by C, then contracted with W_p) would otherwise lose the bits that
// cancel -- the same effect that makes the forward pass carry Y_p as hi + lo; dW_p and dC show it
// in their small entries.
//   dW_p  = dY_p^T X                         r x n,  K = T
//   dC    = dY_np^T Y_p,  Y_p = X W_p^T      (m - r) x r,  K = T    (step 3, reversed)
// M accumulators for one calibration batch (X_o the dense data flow, X_u the low-rank one):
//   Y_t  = (lambda X_o + (1 - lambda) X_u) W^T          T x m   (the mixed target, Eq. 6)
// The mixed input and Y_t are carried as hi + lo bf16 pairs: each feeds a contraction whose sums
// cancel, and a single bf16 rounding of them shows in Y_t X^T's small entries.
//   XXt += X_u^T X_u                                    n x n   (x x^T summed over the batch)
//   YtXt += Y_t^T X_u                                   m x n   (Y_t X^T summed over the batch)
#include <cuda_bf16.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"

namespace {

using namespace pifa;
using bf16 = __nv_bfloat16;

int64_t pad8(int64_t v) { return (v + 7) / 8 * 8; }
int64_t a256(int64_t b) { return (b + 255) / 256 * 256; }

// dY's columns split into its pivot and non-pivot parts (bf16): outp[t][j] = in[t][piv[j]] for
// j < r and outnp[t][i] = in[t][nonpiv[i]] for i < nnp; an index outside [0, bound) writes 0 and
// latches PIFA_ERR_DEVICE_INDEX. A block stages `rows` rows of dY in shared memory with 16-byte
// loads; a thread then owns two neighbouring output columns, reads their indices once and gathers
// them for each staged row into one 4-byte store (both output pitches are multiples of 8 and both
// parts start at even columns). Bound by its 2 x 2 T m bytes; gathering from global memory, one
// 2-byte load and store per element, took 19.1 us for T = 2048, m = 4096, this 12.4 us.
__global__ void __launch_bounds__(256) split_cols(const bf16* in, int64_t ldin, const int32_t* piv, int r,
                                                  const int32_t* nonpiv, int nnp, int bound, int T, int rows, bf16* outp,
                                                  int64_t ldp, bf16* outnp, int64_t ldnp, int* status) {
  extern __shared__ __align__(16) uint16_t row_sm[];  // rows x w, w = bound rounded up to 8
  pdl_launch_dependents();
  pdl_wait_primary();
  const int w = (bound + 7) & ~7, t0 = blockIdx.x * rows, nr = min(rows, T - t0);
  for (int e = threadIdx.x; e < nr * (w / 8); e += 256) {
    const int t = e / (w / 8), c = e - t * (w / 8);
    const bf16* src = in + (int64_t)(t0 + t) * ldin + 8 * c;
    if (8 * c + 8 <= bound) {
      reinterpret_cast<uint4*>(row_sm)[e] = __ldcs(reinterpret_cast<const uint4*>(src));
    } else {
      for (int k = 0; 8 * c + k < bound; ++k) row_sm[8 * e + k] = __bfloat16_as_ushort(src[k]);
    }
  }
  __syncthreads();
  const int np = (r + 1) / 2, nq = (nnp + 1) / 2;  // output pairs of each part
  for (int e = threadIdx.x; e < np + nq; e += 256) {
    const bool pv = e < np;
    const int j = 2 * (pv ? e : e - np), n = pv ? r : nnp;
    const int32_t* idx = (pv ? piv : nonpiv) + j;
    const int c0 = __ldg(idx), c1 = j + 1 < n ? __ldg(idx + 1) : c0;
    const bool ok0 = (unsigned)c0 < (unsigned)bound, ok1 = (unsigned)c1 < (unsigned)bound;
    if (!ok0 || !ok1) latch_status(status, PIFA_ERR_DEVICE_INDEX);
    const int64_t ld = pv ? ldp : ldnp;
    bf16* out = (pv ? outp : outnp) + (int64_t)t0 * ld + j;
#pragma unroll 4
    for (int t = 0; t < nr; ++t) {
      const uint32_t a = ok0 ? row_sm[t * w + c0] : 0u, b = ok1 ? row_sm[t * w + c1] : 0u;
      *reinterpret_cast<uint32_t*>(out + (int64_t)t * ld) = a | b << 16;  // an odd part's last pair ends in its padding
    }
  }
}

// The same straight from global memory, for rows too wide to stage: a thread owns one output column
// and walks the rows of its y-block's share.
__global__ void split_wide(const bf16* in, int64_t ldin, const int32_t* piv, int r, const int32_t* nonpiv, int nnp,
                           int bound, int T, bf16* outp, int64_t ldp, bf16* outnp, int64_t ldnp, int* status) {
  pdl_launch_dependents();
  pdl_wait_primary();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= r + nnp) return;
  const bool pv = j < r;
  const int c = __ldg(pv ? piv + j : nonpiv + (j - r));
  bf16* out = pv ? outp + j : outnp + (j - r);
  const int64_t ldo = pv ? ldp : ldnp;
  const bool ok = (unsigned)c < (unsigned)bound;
  if (!ok) latch_status(status, PIFA_ERR_DEVICE_INDEX);
  const bf16 zero = __float2bfloat16_rn(0.0f);
#pragma unroll 8
  for (int t = blockIdx.y; t < T; t += gridDim.y) out[(int64_t)t * ldo] = ok ? in[(int64_t)t * ldin + c] : zero;
}

// out = a * x + b * y elementwise over T rows of n (bf16 in, fp32 arithmetic), written as a hi +
// lo pair of bf16 planes. A thread owns 8 consecutive columns of a row (16-byte loads and stores:
// every pitch is a multiple of 8 elements and every base 16-byte aligned), scalar at a ragged end.
// Rows across the y grid, column groups across x.
__global__ void axpby_rows(const bf16* x, const bf16* y, int64_t ld, int T, int n, float a, float b, bf16* out,
                           bf16* out_lo, int64_t ldout) {
  pdl_launch_dependents();
  pdl_wait_primary();
  const int ng = (n + 7) / 8;
  for (int t = blockIdx.y; t < T; t += gridDim.y)
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
      const int c = 8 * g;
      const bf16* xr = x + (int64_t)t * ld + c;
      const bf16* yr = y + (int64_t)t * ld + c;
      bf16* hr = out + (int64_t)t * ldout + c;
      bf16* lr = out_lo + (int64_t)t * ldout + c;
      if (c + 8 <= n) {
        uint4 xv = *reinterpret_cast<const uint4*>(xr), yv = *reinterpret_cast<const uint4*>(yr), hv, lv;
        const bf16* xe = reinterpret_cast<const bf16*>(&xv);
        const bf16* ye = reinterpret_cast<const bf16*>(&yv);
        bf16* he = reinterpret_cast<bf16*>(&hv);
        bf16* le = reinterpret_cast<bf16*>(&lv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float v = a * __bfloat162float(xe[e]) + b * __bfloat162float(ye[e]);
          he[e] = __float2bfloat16_rn(v);
          le[e] = __float2bfloat16_rn(v - __bfloat162float(he[e]));
        }
        *reinterpret_cast<uint4*>(hr) = hv;
        *reinterpret_cast<uint4*>(lr) = lv;
      } else {
        for (int e = 0; c + e < n; ++e) {
          const float v = a * __bfloat162float(xr[e]) + b * __bfloat162float(yr[e]);
          const bf16 h = __float2bfloat16_rn(v);
          hr[e] = h;
          lr[e] = __float2bfloat16_rn(v - __bfloat162float(h));
        }
      }
    }
}

// A row-wise elementwise kernel over `rows` rows of `cols` columns: rows on the y grid (at most
// 65535, the kernel loops beyond), columns on x.
int launch_small(const void* fn, void** args, int64_t rows, int64_t cols, cudaStream_t stream, const char* what) {
  cudaLaunchConfig_t cfg = {};
  const int64_t bx = (cols + 255) / 256;
  cfg.gridDim = dim3((unsigned)(bx < 8 ? (bx > 0 ? bx : 1) : 8), (unsigned)(rows < 65535 ? (rows > 0 ? rows : 1) : 65535));
  cfg.blockDim = dim3(256);
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e == cudaSuccess) pifa_count_launch();
  return e == cudaSuccess ? PIFA_OK : pifa_fail_cuda(what, e);
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct BwdLayout {
  int64_t dynp, dyi, yp, yp_lo, dyp, dyp_lo, total;
};

BwdLayout bwd_layout(int64_t T, int64_t m, int64_t r) {
  BwdLayout L;
  int64_t o = 0;
  L.dynp = o;
  o += a256(T * pad8(m - r > 0 ? m - r : 1) * 2);
  L.dyi = o;
  o += a256(T * pad8(r) * 2);
  L.yp = o;
  o += a256(T * pad8(r) * 2);
  L.yp_lo = o;
  o += a256(T * pad8(r) * 2);
  L.dyp = o;
  o += a256(T * pad8(r) * 2);
  L.dyp_lo = o;
  o += a256(T * pad8(r) * 2);
  L.total = o;
  return L;
}

struct MaccLayout {
  int64_t xmix, xmix_lo, ytt, ytt_lo, total;
};

// The mixed input's hi and lo planes (T x pad8(n)), Y_t^T's hi and lo planes (m x pad8(T)), all bf16
MaccLayout macc_layout(int64_t T, int64_t m, int64_t n) {
  MaccLayout L;
  int64_t o = 0;
  L.xmix = o;
  o += a256(T * pad8(n) * 2);
  L.xmix_lo = o;
  o += a256(T * pad8(n) * 2);
  L.ytt = o;
  o += a256(m * pad8(T) * 2);
  L.ytt_lo = o;
  o += a256(m * pad8(T) * 2);
  L.total = o;
  return L;
}

}  // namespace

extern "C" int64_t pifa_backward_workspace_size(int64_t T, int64_t m, int64_t n, int64_t r) {
  pifa_clear_error();
  if (T < 0 || m < 1 || n < 1 || r < 1 || r > m || r > n) return pifa_fail(PIFA_ERR_INVALID_ARG, "need T >= 0 and 1 <= r <= min(m, n)");
  return bwd_layout(T, m, r).total;
}

extern "C" int pifa_backward(const void* X, int64_t T, int64_t n, int64_t ldx, const void* Wp, int64_t r, int64_t ldwp,
                             const void* C, int64_t m, int64_t ldc, const int32_t* pivot_idx,
                             const int32_t* nonpivot_idx, const void* dY, int64_t lddy, void* dX, int64_t lddx,
                             float* dWp, int64_t lddwp, float* dC, int64_t lddc, void* workspace,
                             int64_t workspace_bytes, void* cuda_stream) {
  pifa_clear_error();
  if (T < 0 || m < 1 || n < 1 || r < 1 || r > m || r > n || T >= (1 << 30) || m >= (1 << 30) || n >= (1 << 30))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "need T >= 0 and 1 <= r <= min(m, n) < 2^30");
  const bool has_np = m > r;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (!Wp || !pivot_idx || (has_np && (!C || !nonpivot_idx)))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "null Wp, C, pivot_idx or nonpivot_idx");
  if (ldwp < n || (has_np && ldc < r)) return pifa_fail(PIFA_ERR_INVALID_ARG, "leading dimension smaller than the row");
  if ((dX && lddx < n) || (dWp && lddwp < n) || (dC && lddc < r))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "output leading dimension smaller than the row");
  if (T == 0) {  // no tokens: zero weight gradients
    cudaError_t e = cudaSuccess;
    if (dWp) e = cudaMemset2DAsync(dWp, lddwp * 4, 0, n * 4, r, s);
    if (e == cudaSuccess && dC && has_np) e = cudaMemset2DAsync(dC, lddc * 4, 0, r * 4, m - r, s);
    return e == cudaSuccess ? PIFA_OK : pifa_fail_cuda("backward: zero gradients", e);
  }
  if (!X || !dY) return pifa_fail(PIFA_ERR_INVALID_ARG, "null X or dY");
  if (ldx < n || lddy < m) return pifa_fail(PIFA_ERR_INVALID_ARG, "leading dimension smaller than the row");
  if (!al16(X) || !al16(Wp) || !al16(dY) || (has_np && !al16(C)) || (dX && !al16(dX)) || (dWp && !al16(dWp)) ||
      (dC && !al16(dC)) || ((ldx | ldwp | lddy | (has_np ? ldc : 0) | (dX ? lddx : 0)) & 7) ||
      ((dWp ? lddwp : 0) & 3) || ((dC ? lddc : 0) & 3))
    return pifa_fail(PIFA_ERR_ALIGNMENT, "16-byte aligned buffers and 16-byte row pitches required");
  const BwdLayout Ly = bwd_layout(T, m, r);
  if (!workspace || workspace_bytes < Ly.total) return pifa_fail(PIFA_ERR_WORKSPACE, "workspace missing or too small");
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return pifa_fail(PIFA_ERR_ALIGNMENT, "workspace must be 256-byte aligned");
  cudaError_t ce = cudaSuccess;
  int* status = pifa_status_word(&ce);
  if (!status) return pifa_fail_cuda("device status word", ce);
  const uint64_t tmo = pifa_wait_timeout_ns();
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  bf16* dYnp = reinterpret_cast<bf16*>(ws + Ly.dynp);
  bf16* Yp = reinterpret_cast<bf16*>(ws + Ly.yp);
  bf16* Yp_lo = reinterpret_cast<bf16*>(ws + Ly.yp_lo);
  bf16* dYp = reinterpret_cast<bf16*>(ws + Ly.dyp);
  bf16* dYp_lo = reinterpret_cast<bf16*>(ws + Ly.dyp_lo);
  const int64_t ldnp = pad8(m - r > 0 ? m - r : 1), ldr = pad8(r);
  int st;
  bf16* dYi = reinterpret_cast<bf16*>(ws + Ly.dyi);
  {  // dY_I = dY[:, I] and dY_np = dY[:, I^c] in one pass over dY (dY_I straight into dY_p when r = m)
    cudaLaunchConfig_t cfg = {};
    const int64_t row_bytes = (m + 7) / 8 * 16;
    // rows per block: 72 KB of them (three blocks per SM), or up to three wider ones that share the
    // indices' loads
    int64_t rows = 72 * 1024 / row_bytes;
    if (rows < 3) rows = 200 * 1024 / row_bytes < 3 ? 200 * 1024 / row_bytes : 3;
    if (rows > 16) rows = 16;
    cudaError_t e = cudaSuccess;
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (rows > 0) {
      cfg.gridDim = dim3((unsigned)((T + rows - 1) / rows));
      cfg.dynamicSmemBytes = (size_t)(rows * row_bytes);
      e = cudaFuncSetAttribute(split_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      if (e == cudaSuccess)
        e = pifa_launch_ex(&cfg, split_cols, reinterpret_cast<const bf16*>(dY), lddy, pivot_idx, (int)r, nonpivot_idx,
                           (int)(m - r), (int)m, (int)T, (int)rows, has_np ? dYi : dYp, ldr, dYnp, ldnp, status);
    } else {
      cfg.gridDim = dim3((unsigned)((m + 255) / 256), (unsigned)(T < 64 ? T : 64));
      e = pifa_launch_ex(&cfg, split_wide, reinterpret_cast<const bf16*>(dY), lddy, pivot_idx, (int)r, nonpivot_idx,
                         (int)(m - r), (int)m, (int)T, has_np ? dYi : dYp, ldr, dYnp, ldnp, status);
    }
    if (e != cudaSuccess) return pifa_fail_cuda("backward: split dY", e);
  }
  // Two launches of independent products: those that dY and X give, then those that need them. (One
  // stream per product instead left the last wave of each launch's tiles on a part of the SMs.)
  GemmTc first[2], second[3];
  int n1 = 0, n2 = 0;
  if (has_np) {  // dY_p = dY_I + dY_np C, as hi + lo planes (dY_p = dY_I when r = m)
    GemmTc g = {T, r, m - r, dYnp, ldnp, false, C, ldc, true, dYp, ldr, 3, 1.0f, dYi, ldr};
    g.D2 = dYp_lo;
    first[n1++] = g;
  }
  if (dC && has_np) {  // Y_p = X W_p^T as hi + lo planes (only dC needs it)
    GemmTc g = {T, r, n, X, ldx, false, Wp, ldwp, false, Yp, ldr, 3, 1.0f, nullptr, 0};
    g.D2 = Yp_lo;
    first[n1++] = g;
  }
  if (dX) {  // dX = (dY_p,hi + dY_p,lo) W_p  (dY_p exact in bf16 when r == m)
    GemmTc g = {T, n, r, dYp, ldr, false, Wp, ldwp, true, dX, lddx, 0, 1.0f, nullptr, 0};
    if (has_np) g.A2 = dYp_lo;
    second[n2++] = g;
  }
  if (dWp) {  // dW_p = (dY_p,hi + dY_p,lo)^T X
    GemmTc g = {r, n, T, dYp, ldr, true, X, ldx, true, dWp, lddwp, 1, 1.0f, nullptr, 0};
    if (has_np) g.A2 = dYp_lo;
    second[n2++] = g;
  }
  if (dC && has_np) {  // dC = dY_np^T (Y_p,hi + Y_p,lo)
    GemmTc g = {m - r, r, T, dYnp, ldnp, true, Yp, ldr, true, dC, lddc, 1, 1.0f, nullptr, 0};
    g.B2 = Yp_lo;
    second[n2++] = g;
  }
  if ((st = gemm_tc_group(first, n1, status, tmo, s)) != PIFA_OK) return st;
  return gemm_tc_group(second, n2, status, tmo, s);
}

extern "C" int64_t pifa_m_accumulate_workspace_size(int64_t T, int64_t m, int64_t n) {
  pifa_clear_error();
  if (T < 0 || m < 1 || n < 1) return pifa_fail(PIFA_ERR_INVALID_ARG, "need T >= 0, m >= 1, n >= 1");
  return macc_layout(T, m, n).total;
}

extern "C" int pifa_m_accumulate(const void* Xo, const void* Xu, int64_t T, int64_t n, int64_t ldx, const void* W,
                                 int64_t m, int64_t ldw, float lambda, float* XXt, int64_t ldxx, float* YtXt,
                                 int64_t ldyx, void* workspace, int64_t workspace_bytes, void* cuda_stream) {
  pifa_clear_error();
  if (T < 0 || m < 1 || n < 1 || T >= (1 << 30) || m >= (1 << 30) || n >= (1 << 30))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "need T >= 0 and 1 <= m, n < 2^30");
  if (!(lambda >= 0.0f && lambda <= 1.0f)) return pifa_fail(PIFA_ERR_INVALID_ARG, "lambda must be in [0, 1]");
  if (T == 0) return PIFA_OK;  // nothing to accumulate
  if (!Xu || !XXt || (YtXt && (!W || !Xo))) return pifa_fail(PIFA_ERR_INVALID_ARG, "null Xu, XXt, or W / Xo with YtXt");
  if (ldx < n || ldxx < n || (YtXt && (ldw < n || ldyx < n)))
    return pifa_fail(PIFA_ERR_INVALID_ARG, "leading dimension smaller than the row");
  if (!al16(Xu) || !al16(XXt) || (YtXt && (!al16(Xo) || !al16(W) || !al16(YtXt))) || (ldx & 7) || (ldxx & 3) ||
      (YtXt && ((ldw & 7) || (ldyx & 3))))
    return pifa_fail(PIFA_ERR_ALIGNMENT, "16-byte aligned buffers and 16-byte row pitches required");
  const MaccLayout Ly = macc_layout(T, m, n);
  if (!workspace || workspace_bytes < Ly.total) return pifa_fail(PIFA_ERR_WORKSPACE, "workspace missing or too small");
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return pifa_fail(PIFA_ERR_ALIGNMENT, "workspace must be 256-byte aligned");
  cudaError_t ce = cudaSuccess;
  int* status = pifa_status_word(&ce);
  if (!status) return pifa_fail_cuda("device status word", ce);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  const uint64_t tmo = pifa_wait_timeout_ns();
  int st;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  const int64_t ldT = pad8(T), ldn = pad8(n);
  // XXt += X_u^T X_u, its upper triangle (the product is symmetric: half the tiles)
  GemmTc xx = {n, n, T, Xu, ldx, true, Xu, ldx, true, XXt, ldxx, 2, 1.0f, nullptr, 0};
  xx.upper = true;
  if (!YtXt) return gemm_tc_group(&xx, 1, status, tmo, s);
  bf16* Xmix = reinterpret_cast<bf16*>(ws + Ly.xmix);
  bf16* Xmix_lo = reinterpret_cast<bf16*>(ws + Ly.xmix_lo);
  bf16* YtT = reinterpret_cast<bf16*>(ws + Ly.ytt);
  bf16* YtT_lo = reinterpret_cast<bf16*>(ws + Ly.ytt_lo);
  {  // X_mix = lambda X_o + (1 - lambda) X_u, as hi + lo planes
    int Ti = (int)T, ni = (int)n;
    float a = lambda, b = 1.0f - lambda;
    void* args[] = {(void*)&Xo, (void*)&Xu, (void*)&ldx, (void*)&Ti, (void*)&ni, (void*)&a, (void*)&b, (void*)&Xmix,
                    (void*)&Xmix_lo, (void*)&ldn};
    if ((st = launch_small((const void*)axpby_rows, args, T, (n + 7) / 8, s, "m_accumulate: mix")) != PIFA_OK) return st;
  }
  // Y_t^T = W (X_mix,hi + X_mix,lo)^T, as hi + lo planes (m x T), beside X X^T, whose tiles fill the
  // SMs that Y_t^T's last wave leaves; then YtXt += (Y_t^T,hi + Y_t^T,lo) X_u
  GemmTc yt = {m, T, n, W, ldw, false, Xmix, ldn, false, YtT, ldT, 3, 1.0f, nullptr, 0};
  yt.B2 = Xmix_lo;
  yt.D2 = YtT_lo;
  GemmTc yx = {m, n, T, YtT, ldT, false, Xu, ldx, true, YtXt, ldyx, 2, 1.0f, nullptr, 0};
  yx.A2 = YtT_lo;
  const GemmTc first[2] = {yt, xx};
  if ((st = gemm_tc_group(first, 2, status, tmo, s)) != PIFA_OK) return st;
  return gemm_tc_group(&yx, 1, status, tmo, s);
}
