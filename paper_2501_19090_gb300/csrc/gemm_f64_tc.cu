// gemm_f64_tc.cu -- float64 matrix products on the 5th-generation tensor cores, by exact slices,
// for the float64 set-up paths (Algorithm 1 and the M reconstruction's solves).
//
// sm_103a issues about two float64 multiply-adds per clock and SM (1.1 TFLOP/s measured with the
// CUDA-core gemm_f64), against 4096 bf16 ones, so a float64 product is computed as integers (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, 2012): every row of A and column of B is
// scaled by a power of two to below one in magnitude, rounded to 62 fractional bits (float64 keeps
// 53 of its own), and cut into 8 balanced base-256 digits, each a whole number of at most 8 bits
// and so exact in bf16. With a_p, b_q the digit matrices,
//   A B = sum over d = p + q <= 7 of 2^-(12 + 8 d) V_d,   V_d = sum over p + q = d of a_p b_q.
// A V_d over K = 128 columns is a whole number of at most 8 128 128^2 = 2^24, which the fp32 accumulators
// in tensor memory hold exactly; every 128 columns the 8 accumulators are drained into 64-bit integers.
// Beside the final rounding to float64, element (i, j) is off by the operands' rounding and the dropped
// pairs (d > 7). With A_i and B_j the scales of row i and column j (powers of two above their largest
// magnitudes) that is at most 2^-59 A_i B_j per term (seven pairs d = 8 of up to 2^14 2^-76, and 2^-62),
// and 2^-62.2 A_i B_j sqrt(K) in the root mean square. The bound is relative to the largest entries, not to
// the terms themselves: where small entries meet large ones, or one entry of a row towers above the
// others, a chain of float64 multiply-adds, off by up to K 2^-53 S_ij with S_ij = sum over k of |a_ik b_kj|,
// can be far better. So the elements with S_ij < sqrt(K) / 128 A_i B_j (K: the terms that triangular
// operands leave) are computed by such a chain, in the order of the CUDA-core products; the others are off
// by at most 2 sqrt(K) 2^-53 S_ij, and by 0.22 2^-53 S_ij in the root mean square, less than one rounding.
// S comes from the operands' magnitudes in bf16 (truncated, and not below 2^-60, so that S = 0 means that
// every term is zero), one more product of bf16 matrices (gemm_tc.cu) whose epilogue writes a bit per
// element: 1 / 36 of the digits' multiply-adds. Products with themselves (A = B^T) need none: theirs enter
// or leave a Cholesky factorisation, whose own error in element (i, j) is a multiple of 2^-53 times the
// geometric mean of the diagonal elements i and j, each at least its scale's square over four.
// Against quad precision W_p = U V^T (K = 256 to 2048, N(0, 1) factors) is 4.7e-17 off, its float64
// rounding, where the chain is 5e-16 to 1.1e-15 off; so it is with U D and V / D for any diagonal D of powers
// of two, for which slices alone lose all digits at D = 2^-30 to 2^30.
//
// Sliced operands are laid out [row][K block of 32][digit][32], so that a TMA box of 64 elements
// holds two digits of one K block as one 128-byte swizzled row.
//
// One CTA per 128 x 64 output tile, 320 threads: warp 0 the TMA producer (two 96 KB stages of one K
// block: 8 digits of 128 rows of A and 64 of B), warp 1 the MMA issuer (accumulators d = 0 .. 7 of 64
// columns: all 512 columns of tensor memory; a digit of A times up to four digits of B in one
// instruction of M = 128, N = 64 to 256, K = 16: 30 instructions a stage for the 36 digit pairs), warps
// 2-9 the drain. In the last stage of a K = 128 chunk accumulator i is complete, and committed by
// itself, after A's digit i, so that most of the drain runs under the chunk's own MMAs. Every wait is
// bounded. 2048 x 2048 x 2048: 645 -> 302 us against one N = 64 instruction per pair (each 66 cycles, of
// which its multiply-adds are 33), 2.0 PFLOP/s of the tensor cores; feeding those from a pair of CTAs
// changed nothing (641).
#include <cuda_bf16.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"

namespace {

using namespace pifa;

constexpr int SM_ = 128, SN = 64;        // output tile
constexpr int KBLK = 32;                 // K columns per stage
constexpr int NDIG = 8;                  // digits per value, and diagonals kept
constexpr int CHUNK = 4;                 // stages per exact accumulation: 128 columns of K
constexpr int ROWLEN = KBLK * NDIG;      // sliced elements per row and K block
constexpr uint32_t A_BOX = SM_ * 128, B_BOX = SN * 128;  // two digits: 128-byte rows
constexpr uint32_t STAGE = (NDIG / 2) * (A_BOX + B_BOX);
constexpr int STAGES = 2;
constexpr int DRAIN_WARPS = 8;
constexpr int THREADS = 64 + 32 * DRAIN_WARPS;
constexpr size_t SMEM = 1024 + STAGES * STAGE + 256;
constexpr uint32_t TMEM_COLS = NDIG * SN;  // 512
// Columns of K per panel: the drain adds up to 2^24 2^24 = 2^48 to a 64-bit sum for every 128 of them
// (V_4 and V_0 shifted by 24 bits, the others by less).
constexpr int64_t kMaxPanel = (int64_t)1 << 20;
static_assert(kMaxPanel / (KBLK * CHUNK) <= ((int64_t)1 << 14), "the drain's sums stay below 2^62");
// First column of accumulator d: the even ones, then the odd ones (see the MMA issuer).
__host__ __device__ constexpr uint32_t acc_col(int d) { return (uint32_t)((d & 1) * (NDIG / 2) + (d >> 1)) * SN; }

// ---- slicing -----------------------------------------------------------------------------------
struct SliceArgs {
  const double* X;     // element (i, k) at X[row(i) * s_row + k * s_k], row(i) = idx ? idx[i] : i
  const int32_t* idx;
  int64_t s_row, s_k;
  int rows, K;
  unsigned long long* mx;   // per row: the bits of max |x| over k
  __nv_bfloat16* S;         // rows x (nkb ROWLEN)
  int nkb;
  __nv_bfloat16* mag;       // rows x (nkb KBLK): the magnitudes over the row's scale (null: not needed)
};

// max |x| of each row as an unsigned bit pattern (non-negative float64 values order like their
// bits, and every NaN and infinity orders above the finite ones). mx must be zero on entry.
__global__ void __launch_bounds__(256) slice_row_max(SliceArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = blockIdx.x * 32;
  const int per = (a.K + gridDim.y - 1) / gridDim.y;
  const int k0 = blockIdx.y * per, k1 = min(a.K, k0 + per);
  if (a.s_k == 1) {  // the lanes along K; a warp takes 4 of the block's 32 rows
    for (int rr = warp; rr < 32; rr += 8) {
      const int i = r0 + rr;
      if (i >= a.rows) continue;
      const double* x = a.X + (a.idx ? (int64_t)a.idx[i] : (int64_t)i) * a.s_row;
      unsigned long long m = 0;
#pragma unroll 4
      for (int k = k0 + lane; k < k1; k += 32)
        m = max(m, (unsigned long long)__double_as_longlong(x[k]) & 0x7fffffffffffffffull);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) atomicMax(a.mx + i, m);
    }
  } else {  // the lanes along the rows; the warps along K
    const int i = r0 + lane;
    if (i >= a.rows) return;
    const double* x = a.X + (a.idx ? (int64_t)a.idx[i] : (int64_t)i) * a.s_row;
    unsigned long long m = 0;
#pragma unroll 4
    for (int k = k0 + warp; k < k1; k += 8)
      m = max(m, (unsigned long long)__double_as_longlong(x[(int64_t)k * a.s_k]) & 0x7fffffffffffffffull);
    atomicMax(a.mx + i, m);
  }
}

// The biased exponent of a row's scale: |x| < 2^(e - 1022) for every x of the row (1 for rows of
// zeros and subnormals, 2047 for a row that holds an infinity or a NaN).
__device__ __forceinline__ int row_exp(unsigned long long mx) {
  const int e = (int)(mx >> 52);
  return e < 1 ? 1 : e;
}

// (hi 2^-36 + lo 2^-68) 2^e rounded to the nearest float64 (ties to even), in integer arithmetic: a
// float64 instruction costs an SM as much issue time as some 30 integer ones.
__device__ __forceinline__ double fixed_to_f64(long long hi, long long lo, int e) {
  unsigned long long l = ((unsigned long long)hi << 32) + (unsigned long long)lo;  // hi 2^32 + lo, 128 bits
  long long h = (hi >> 32) + (lo >> 63) + (l < (unsigned long long)lo ? 1 : 0);
  const bool neg = h < 0;
  if (neg) {
    l = ~l + 1ull;
    h = ~h + (l == 0ull ? 1 : 0);
  }
  unsigned long long m = (unsigned long long)h, rest = l;
  int ex = 127;
  if (m == 0ull) {
    m = l;
    rest = 0ull;
    ex = 63;
  }
  if (m == 0ull) return 0.0;
  const int lz = __clzll((long long)m);
  ex -= lz;
  if (lz) {
    m = (m << lz) | (rest >> (64 - lz));
    rest <<= lz;
  }
  const unsigned int low = (unsigned int)m & 0x7ffu;
  m >>= 11;  // 53 bits
  if (low > 0x400u || (low == 0x400u && (rest != 0ull || (m & 1ull)))) ++m;
  const int be = ex - 68 + e + 1023;
  double v;
  if (be > 1 && be < 2045)
    v = __longlong_as_double((long long)(((unsigned long long)(be - 1) << 52) + m));
  else
    v = scalbn((double)m, be - 1023 - 52);
  return neg ? -v : v;
}

// The 8 digits of one 32 x 32 block of values per CTA of 128 threads: loaded with the lanes along
// the contiguous index, then 4 threads a row, 8 values and 8 x 16 bytes of digits each.
__global__ void __launch_bounds__(128) slice_digits(SliceArgs a) {
  __shared__ unsigned long long t[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = blockIdx.y * 32, kb = blockIdx.x, k0 = kb * KBLK;
  for (int u = warp; u < 32; u += 4) {
    const int rr = a.s_k == 1 ? u : lane, kk = a.s_k == 1 ? lane : u;
    const int i = r0 + rr, k = k0 + kk;
    double x = 0.0;
    if (i < a.rows && k < a.K) x = a.X[(a.idx ? (int64_t)a.idx[i] : (int64_t)i) * a.s_row + (int64_t)k * a.s_k];
    t[rr][kk] = (unsigned long long)__double_as_longlong(x);
  }
  __syncthreads();
  const int rr = threadIdx.x >> 2, kq = (threadIdx.x & 3) * 8;
  const int i = r0 + rr;
  if (i >= a.rows) return;
  const int er = row_exp(a.mx[i]);
  uint32_t w[NDIG][4];  // 8 bf16 digits per plane, packed in pairs
  uint32_t mg[4];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned long long b = t[rr][kq + e];
    int ex = (int)((b >> 52) & 2047);
    unsigned long long mant = b & 0xfffffffffffffull;
    if (ex) mant |= 0x10000000000000ull;
    else ex = 1;
    const int sh = ex - er + 9;  // mant 2^sh = |x| 2^62 / 2^(er - 1022)
    unsigned long long mag = 0;
    if (sh >= 0) mag = mant << sh;  // sh <= 9: ex <= er
    else if (sh > -60) mag = (mant + (1ull << (-sh - 1))) >> -sh;
    if (er == 2047) mag = 0;  // the drain computes this row by plain_dot
    // |x| / 2^(er - 1022) = mant 2^(ex - er - 53), truncated to bf16; at least 2^-60 unless x = 0
    float f = __uint2float_rz((uint32_t)(mant >> 22)) * __uint_as_float((uint32_t)max(ex - er - 31 + 127, 1) << 23);
    f = mant == 0ull || er == 2047 ? 0.0f : fmaxf(f, 0x1p-60f);
    if (e & 1) mg[e >> 1] |= __float_as_uint(f) & 0xffff0000u;
    else mg[e >> 1] = __float_as_uint(f) >> 16;
    long long q = (b >> 63) ? -(long long)mag : (long long)mag;
#pragma unroll
    for (int p = NDIG - 1; p >= 0; --p) {
      const int d = p > 0 ? (int)(signed char)(q & 255) : (int)q;
      q = (q - d) >> 8;
      const uint32_t h = __float_as_uint((float)d) >> 16;  // |d| <= 128: exact in bf16
      if (e & 1) w[p][e >> 1] |= h << 16;
      else w[p][e >> 1] = h;
    }
  }
  __nv_bfloat16* s = a.S + (int64_t)i * a.nkb * ROWLEN + (int64_t)kb * ROWLEN + kq;
#pragma unroll
  for (int p = 0; p < NDIG; ++p) *reinterpret_cast<uint4*>(s + p * KBLK) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
  if (a.mag) *reinterpret_cast<uint4*>(a.mag + ((int64_t)i * a.nkb + kb) * KBLK + kq) = make_uint4(mg[0], mg[1], mg[2], mg[3]);
}

// ---- the products --------------------------------------------------------------------------------
struct SplitArgs {
  int M, N, kbase, K;  // this panel's columns [kbase, kbase + K) of the contraction
  SliceArgs a, b;      // the panel's operands before slicing
  int tri, lower, first;
  double* C;
  const int32_t* cidx;
  int64_t ldc;
  int64_t zc;  // elements between the partial results of consecutive K-slices (blockIdx.z)
  double alpha, beta;
  const uint32_t* mask;  // the elements to leave alone, a bit each (null: none); gemm_f64_flagged computes them
  int words;             // its pitch
  int* status;
  uint64_t timeout_ns;
};

// Element (i, j) over the panel's columns [k0, k1) by float64 multiply-adds: rows and columns that hold
// an infinity or a NaN have no slices, and which elements they turn into which of the two is for the
// arithmetic to say.
__device__ __noinline__ double plain_dot(const SliceArgs& a, const SliceArgs& b, int i, int j, int k0, int k1) {
  const double* x = a.X + (a.idx ? (int64_t)a.idx[i] : (int64_t)i) * a.s_row;
  const double* y = b.X + (b.idx ? (int64_t)b.idx[j] : (int64_t)j) * b.s_row;
  double s = 0.0;
  for (int k = k0; k < k1; ++k) s = fma(x[(int64_t)k * a.s_k], y[(int64_t)k * b.s_k], s);
  return s;
}

__global__ void __launch_bounds__(THREADS, 1)
    gemm_f64_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, SplitArgs p) {
  const int m0 = blockIdx.y * SM_, n0 = blockIdx.x * SN;
  if (p.lower && n0 > m0 + SM_ - 1) return;  // tile wholly above the diagonal
  // columns of K that can hold anything (triangular operands), as stages of this panel
  int ka = 0, ke = p.kbase + p.K;
  if (p.tri & 1) ka = max(ka, n0);
  if (p.tri & 4) ka = max(ka, m0);
  if (p.tri & 2) ke = min(ke, n0 + SN);
  const int kb0 = max(0, ka - p.kbase) / KBLK, kb1 = ke > p.kbase ? (ke - p.kbase + KBLK - 1) / KBLK : 0;
  const int nall = max(0, kb1 - kb0);
  // this K-slice's stages (whole chunks, so that the last one of a slice is not cut short)
  const int per = ((nall + CHUNK - 1) / CHUNK + (int)gridDim.z - 1) / (int)gridDim.z * CHUNK;
  const int sb0 = kb0 + min(nall, (int)blockIdx.z * per), nst = min(nall, ((int)blockIdx.z + 1) * per) - (sb0 - kb0);
  if (nst == 0 && !p.first) return;
  double* const Cz = p.C + blockIdx.z * p.zc;
  const int nch = (nst + CHUNK - 1) / CHUNK;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint64_t* acce = accf + NDIG;
  uint64_t* done = acce + NDIG;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int d = 0; d < NDIG; ++d) {
      mbar_init(&accf[d], 1);
      mbar_init(&acce[d], DRAIN_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int it = 0; it < nst; ++it) {
        const int s = it % STAGES;
        if ((it >= STAGES && !mbar_wait(&empty[s], (uint32_t)((it / STAGES) - 1) & 1u, p.timeout_ns)) || *abort_flag) {
          latch_status(p.status, PIFA_ERR_TIMEOUT);
          *abort_flag = 1;
          break;
        }
        uint8_t* sa = smem + s * STAGE;
        uint8_t* sb = sa + (NDIG / 2) * A_BOX;
        const int x = (sb0 + it) * ROWLEN;
        mbar_arrive_expect_tx(&full[s], STAGE);
        for (int q = 0; q < NDIG / 2; ++q) {
          tma_load_2d(smem_u32(sa + q * A_BOX), &tmA, x + 64 * q, m0, &full[s]);
          tma_load_2d(smem_u32(sb + q * B_BOX), &tmB, x + 64 * q, n0, &full[s]);
        }
        issued = it + 1;
      }
      for (int i = issued > STAGES ? issued - STAGES : 0; i < issued; ++i)
        if (!mbar_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u, 100000000ull))
          latch_status(p.status, PIFA_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // A digit i times the even digits of B is one MMA: box q of B holds digits 2 q and 2 q + 1 side by
      // side, so every second digit is 64 rows further on, and accumulators i, i + 2, .. are
      // adjacent columns; and so the odd digits. An MMA costs at least the 64 cycles of reading its
      // 128 rows of A: 36 pairs one by one took twice the time of their multiply-adds.
      bool dead = false;
      for (int it = 0; it < nst && !dead; ++it) {
        const int s = it % STAGES, ch = it / CHUNK, w = it % CHUNK;
        const bool last = w == CHUNK - 1 || it == nst - 1;
        if (!mbar_wait(&full[s], (uint32_t)(it / STAGES) & 1u, p.timeout_ns) || *abort_flag) {
          dead = true;
          break;
        }
        tc_fence_after();
        const uint32_t a = smem_u32(smem + s * STAGE), b = a + (NDIG / 2) * A_BOX;
        for (int d = 0; w == 0 && ch > 0 && d < NDIG; ++d)  // the drain has taken the last chunk
          if (!mbar_wait(&acce[d], (uint32_t)(ch - 1) & 1u, p.timeout_ns)) {
            dead = true;
            break;
          }
        if (dead) break;
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < NDIG; ++i) {
          const uint32_t pa = a + (uint32_t)(i >> 1) * A_BOX + (uint32_t)(i & 1) * 64u;
          const uint32_t even = idesc_bf16_f32(SM_, SN * ((NDIG + 1 - i) / 2)), odd = idesc_bf16_f32(SM_, SN * ((NDIG - i) / 2));
#pragma unroll
          for (int kk = 0; kk < KBLK / 16; ++kk) {
            const uint32_t acc = (w > 0 || i > 0 || kk > 0) ? 1u : 0u;
            mma_bf16_ss(tmem + acc_col(i), sw128_desc(pa + kk * 32), sw128_desc(b + kk * 32), even, acc);
            if (i + 1 < NDIG)
              mma_bf16_ss(tmem + acc_col(i + 1), sw128_desc(pa + kk * 32), sw128_desc(b + 64u + kk * 32), odd, acc);
          }
          if (last) mma_commit(&accf[i]);  // accumulator i has no terms of the later digits of A
        }
        mma_commit(&empty[s]);
      }
      if (dead) {
        latch_status(p.status, PIFA_ERR_TIMEOUT);
        *abort_flag = 1;
      }
      mma_commit(done);
      if (!mbar_wait(done, 0, 100000000ull)) latch_status(p.status, PIFA_ERR_TIMEOUT);
    }
  } else {
    // drain: TMEM lane quarter warp % 4, 32 of the tile's 64 columns
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    long long hi[32], lo[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
    bool ok = true;
    for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
      for (int d = 0; d < NDIG; ++d) {
        if (ok && !mbar_wait(&accf[d], (uint32_t)ch & 1u, p.timeout_ns)) {
          latch_status(p.status, PIFA_ERR_TIMEOUT);
          *abort_flag = 1;
          ok = false;
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        uint32_t v[32];
        tmem_ld_32x32b_x32(tmem + ((uint32_t)(q4 * 32) << 16) + acc_col(d) + (uint32_t)(half * 32), v);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[d]);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const long long x = (long long)__float2int_rn(__uint_as_float(v[c]));
          if (d < 4) hi[c] += x * (1ll << (8 * (3 - d)));
          else lo[c] += x * (1ll << (8 * (7 - d)));
        }
      }
      if (!ok) break;
    }
    // through shared memory (the ring: every MMA has completed and no copy is in flight once the
    // last accumulator is full), so that the lanes store consecutive columns
    if (ok) {
      fence_proxy_async_smem();
      double* tile = reinterpret_cast<double*>(smem) + (warp - 2) * 32 * 33;
      const int j = n0 + half * 32 + lane, r0 = m0 + q4 * 32, nr = min(32, p.M - r0);
      const bool jn = j < p.N;
      const int ea = lane < nr ? row_exp(p.a.mx[r0 + lane]) : 1, eb = jn ? row_exp(p.b.mx[j]) : 1;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const int e2 = __shfl_sync(0xffffffffu, eb, c);
        tile[lane * 33 + c] = fixed_to_f64(hi[c], lo[c], ea + e2 - 2044);
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, ea == 2047 || eb == 2047)) {
        const int kc = (p.tri & 4) ? ((r0 & ~63) - p.kbase) : 0;  // a triangular A: from its rows' block of 64 on
        const int c0 = max(sb0 * KBLK, kc), c1 = min(p.K, min((sb0 + nst) * KBLK, ke - p.kbase));
        for (int g = 0; g < nr; ++g) {
          const int e1 = __shfl_sync(0xffffffffu, ea, g);
          if (jn && (e1 == 2047 || eb == 2047)) tile[g * 33 + lane] = plain_dot(p.a, p.b, r0 + g, j, c0, c1);
        }
      }
      const bool neg = p.alpha == -1.0, one = neg || p.alpha == 1.0;
      const uint32_t skip = p.mask && lane < nr && n0 + half * 32 < p.N
                                ? p.mask[(int64_t)(r0 + lane) * p.words + (n0 >> 5) + half] : 0u;
      double* c = Cz + (int64_t)r0 * p.ldc + (jn ? (p.cidx ? (int64_t)p.cidx[j] : (int64_t)j) : 0);
      for (int g8 = 0; g8 < nr; g8 += 8) {
        double old[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) old[u] = p.beta != 0.0 && jn && g8 + u < nr ? c[(int64_t)(g8 + u) * p.ldc] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t sk = __shfl_sync(0xffffffffu, skip, g8 + u);
          if (!jn || g8 + u >= nr || (sk >> lane & 1u)) continue;
          double v = tile[(g8 + u) * 33 + lane];
          if (!one) v *= p.alpha;
          else if (neg) v = -v;
          if (p.beta != 0.0) v += p.beta == 1.0 ? old[u] : p.beta * old[u];
          c[(int64_t)(g8 + u) * p.ldc] = v;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

int64_t a1k(int64_t b) { return (b + 1023) / 1024 * 1024; }
constexpr float kLeast = 1.0f / 128.0f;  // S_ij / (A_i B_j sqrt(K)) below which an element is recomputed

bool with_itself(const GemmF64& p) {
  return p.A == p.B && p.sa_i == p.sb_j && p.sa_k == p.sb_k && p.M == p.N && !p.aidx;
}
bool checked(const GemmF64& p) { return !with_itself(p) && !p.normwise; }
int mask_words(const GemmF64& p) { return (p.N + 31) / 32; }

// scratch bytes of a product's sliced operands, their magnitudes and the mask over a panel of kp columns
int64_t panel_bytes(const GemmF64& p, int64_t kp) {
  const int64_t nkb = (kp + KBLK - 1) / KBLK, row = nkb * ROWLEN * 2, mag = checked(p) ? nkb * KBLK * 2 : 0;
  return a1k(p.M * row) + a1k(p.M * 8ll) + a1k(p.M * mag) +
         (with_itself(p) ? 0 : a1k(p.N * row) + a1k(p.N * 8ll) + a1k(p.N * mag)) +
         (checked(p) ? a1k((int64_t)p.M * mask_words(p) * 4) : 0);
}

int slice(const SliceArgs& a, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.mx, 0, (size_t)a.rows * 8, s);
  if (e != cudaSuccess) return pifa_fail_cuda("f64 slices: memset", e);
  const int rb = (a.rows + 31) / 32;
  int ks = 608 / rb;
  if (ks > (a.K + 127) / 128) ks = (a.K + 127) / 128;
  if (ks < 1) ks = 1;
  slice_row_max<<<dim3((unsigned)rb, (unsigned)ks), 256, 0, s>>>(a);
  pifa_count_launch();
  slice_digits<<<dim3((unsigned)a.nkb, (unsigned)rb), 128, 0, s>>>(a);
  pifa_count_launch();
  e = cudaGetLastError();
  return e == cudaSuccess ? PIFA_OK : pifa_fail_cuda("f64 slices: launch", e);
}

}  // namespace

bool gemm_f64_split_fits(const GemmF64& p, int64_t bytes) {
  const int64_t work = (int64_t)p.M * p.N * p.K;
  return p.K >= 64 && work >= (int64_t)1 << 20 && (p.M + 31) / 32 <= 65535 && (p.N + 31) / 32 <= 65535 &&
         panel_bytes(p, p.K < 128 ? p.K : 128) <= bytes - 256;  // 256: alignment of the scratch
}

int gemm_f64_split(const GemmF64& p, void* scratch, int64_t bytes, cudaStream_t stream, int slices, int64_t zc) {
  cudaError_t e = cudaSuccess;
  int* status = pifa_status_word(&e);
  if (!status) return pifa_fail_cuda("device status word", e);
  const int64_t shift = (int64_t)((256 - (reinterpret_cast<uintptr_t>(scratch) & 255u)) & 255u);
  scratch = static_cast<uint8_t*>(scratch) + shift;
  bytes -= shift;
  const bool same = with_itself(p), check = checked(p);
  if (check && slices > 1) return pifa_fail(PIFA_ERR_INVALID_ARG, "gemm_f64_split: a checked product in K-slices");
  int64_t kp = p.K;  // the widest panel of whole 128-column chunks that fits the scratch and the drain's sums
  if (kp > kMaxPanel || panel_bytes(p, kp) > bytes) {
    kp = kp > kMaxPanel ? kMaxPanel : (kp + 127) / 128 * 128;
    while (kp > 128 && panel_bytes(p, kp) > bytes) kp -= 128;
  }
  e = cudaFuncSetAttribute(gemm_f64_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return pifa_fail_cuda("cudaFuncSetAttribute(gemm_f64_split)", e);
  for (int64_t k0 = 0; k0 < p.K; k0 += kp) {
    const int kn = (int)(p.K - k0 < kp ? p.K - k0 : kp);
    const int nkb = (kn + KBLK - 1) / KBLK;
    const int64_t row = (int64_t)nkb * ROWLEN * 2;
    uint8_t* w = static_cast<uint8_t*>(scratch);
    auto take = [&](int64_t n) {
      uint8_t* at = w;
      w += a1k(n);
      return at;
    };
    const int64_t mag = (int64_t)nkb * KBLK * 2;
    SliceArgs a = {p.A + k0 * p.sa_k, p.aidx, p.sa_i, p.sa_k, p.M, kn, nullptr, nullptr, nkb, nullptr};
    a.S = reinterpret_cast<__nv_bfloat16*>(take(p.M * row));
    a.mx = reinterpret_cast<unsigned long long*>(take((int64_t)p.M * 8));
    if (check) a.mag = reinterpret_cast<__nv_bfloat16*>(take(p.M * mag));
    SliceArgs b = a;
    int st = slice(a, stream);
    if (st != PIFA_OK) return st;
    if (!same) {
      b = SliceArgs{p.B + k0 * p.sb_k, nullptr, p.sb_j, p.sb_k, p.N, kn, nullptr, nullptr, nkb, nullptr};
      b.S = reinterpret_cast<__nv_bfloat16*>(take(p.N * row));
      b.mx = reinterpret_cast<unsigned long long*>(take((int64_t)p.N * 8));
      if (check) b.mag = reinterpret_cast<__nv_bfloat16*>(take(p.N * mag));
      if ((st = slice(b, stream)) != PIFA_OK) return st;
    }
    uint32_t* mask = nullptr;
    const int words = mask_words(p);
    if (check) {  // one bit per element: S_ij < kLeast sqrt(terms), S in units of A_i B_j
      mask = reinterpret_cast<uint32_t*>(take((int64_t)p.M * words * 4));
      GemmTc c = {p.M, p.N, kn, a.mag, mag / 2, false, b.mag, mag / 2, false, mask, words, 4, kLeast, nullptr, 0};
      c.tri = p.tri;
      c.k0 = (int)k0;
      c.k1 = (int)k0 + kn;
      if ((st = gemm_tc_group(&c, 1, status, pifa_wait_timeout_ns(), stream)) != PIFA_OK) return st;
    }
    CUtensorMap tA, tB;
    if ((st = make_tmap_2d(&tA, PIFA_DTYPE_BF16, a.S, p.M, row / 2, row / 2, 64, SM_)) != PIFA_OK) return st;
    if ((st = make_tmap_2d(&tB, PIFA_DTYPE_BF16, b.S, p.N, row / 2, row / 2, 64, SN)) != PIFA_OK) return st;
    SplitArgs g = {};
    g.M = p.M;
    g.N = p.N;
    g.kbase = (int)k0;
    g.K = kn;
    g.tri = p.tri;
    g.lower = p.lower;
    g.first = k0 == 0;
    g.a = a;
    g.b = b;
    g.C = p.C;
    g.cidx = p.cidx;
    g.ldc = p.ldc;
    g.alpha = p.alpha;
    g.beta = k0 == 0 ? p.beta : 1.0;
    g.zc = zc;
    g.mask = mask;
    g.words = words;
    g.status = status;
    g.timeout_ns = pifa_wait_timeout_ns();
    const dim3 grid((unsigned)((p.N + SN - 1) / SN), (unsigned)((p.M + SM_ - 1) / SM_), (unsigned)slices);
    if (grid.y > 65535u) return pifa_fail(PIFA_ERR_UNSUPPORTED, "gemm_f64_split: more than 65535 row tiles");
    gemm_f64_split_kernel<<<grid, THREADS, SMEM, stream>>>(tA, tB, g);
    e = cudaGetLastError();
    if (e != cudaSuccess) return pifa_fail_cuda("gemm_f64_split launch", e);
    pifa_count_launch();
    if (check) {
      GemmF64 f = p;
      f.A += k0 * p.sa_k;
      f.B += k0 * p.sb_k;
      f.K = kn;
      f.kbase = (int)k0;
      f.beta = g.beta;
      if ((st = gemm_f64_flagged(f, mask, words, stream)) != PIFA_OK) return st;
    }
  }
  return PIFA_OK;
}
