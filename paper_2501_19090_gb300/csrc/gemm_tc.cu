// gemm_tc.cu -- general bf16 contractions D = alpha A B^T (+ addend) on the 5th-generation tensor
// cores, for the PIFA backward pass (fine-tuning, Sec. 5.1; Sec. 6) and the M online accumulators
// (Sec. 4): products whose operands are stored transposed (MN-major).
//
//   A is M x K, B is N x K (bf16). Each operand is either K-major (stored as rows of K contiguous
//   elements: A[m * lda + k]) or MN-major (stored as K rows of contiguous M or N: A[k * lda + m]);
//   the instruction descriptor's transpose bits tell the tensor core which, and TMA fetches
//   K-major tiles as 128 x 64 boxes and MN-major tiles as 64 (MN) x 64 (K) boxes, 128-byte swizzle.
//   D (M x N, fp32 accumulate) is written as bf16, as fp32, added into an fp32 matrix, or as a
//   hi + lo pair of bf16 matrices (hi = bf16(D), lo = bf16(D - hi)) for a later contraction that must
//   not lose D's low bits. A second K pass into the same accumulator with A2 in place of A and/or
//   B2 in place of B (same layouts) consumes such a pair: D = (A + A2) B^T or A (B + B2)^T. For the sliced
//   float64 products D can also be one bit per element, whether it is small against its terms.
//
// One launch computes up to three independent products on a persistent grid of CTA pairs (clusters of
// two, one CTA of 352 threads per SM). A pair computes 256 x bn tiles (bn <= 256) with pair MMAs
// (cta_group::2: M = 256, N = bn, K = 16): each CTA loads its 128 rows of A and half of B's rows, 32 KB
// per 64 columns of K instead of 48 KB, into a 6-stage ring that runs on from tile to tile (warp 0
// loads A, the last warp B); the even CTA's warp 1 issues the MMAs of both into one of two
// accumulators (256 TMEM columns each); warps 2-9 of each CTA drain the other one meanwhile, so that
// the conversions, the values to add in and the stores of a tile run under the next tile's MMAs.
// The main loop is bound by the threads that issue: a flag read from shared memory per step, the
// stage index by division and the MN-major boxes in a loop cost it up to 45%. Measured, K-major,
// 4864 x 4096 x 8192 (four whole rounds of tiles): 1925 TFLOP/s, cuBLAS's burst rate; 4096 x 4096,
// r = 2048, T = 2048: backward 316.5 -> 164 to 170 us and the M accumulators of two batches 860 ->
// 440 us against the form that this replaced (a launch and a CTA per tile of up to 128 x 256 with
// the epilogue exposed, products on side streams), every output bit for bit the same; one-CTA MMAs
// on the same persistent grid took 253.6 and 538.1 us.
// Every wait is bounded (globaltimer); on timeout the CTA latches PIFA_ERR_TIMEOUT, drains what it
// has in flight and returns.
#include <map>
#include <mutex>

#include <cuda_bf16.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"

namespace {

using namespace pifa;
using bf16 = __nv_bfloat16;

constexpr int BM = 128;       // rows of one CTA; a pair of CTAs computes 256 x bn tiles
constexpr int PM = 2 * BM;
constexpr int BNMAX = 256;
constexpr int BK = 64;
constexpr int STAGES = 6;
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 96 + 32 * EPI_WARPS;
constexpr uint32_t A_BYTES = BM * BK * 2;             // 16 KB
constexpr uint32_t STAGE_BYTES = A_BYTES + BNMAX / 2 * BK * 2;  // this CTA's halves of the pair's tiles
constexpr uint32_t MN_BOX = 64 * BK * 2;              // one MN-major box: 64 (MN) x 64 (K), 8 KB
constexpr size_t SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + 256;
constexpr uint32_t TMEM_COLS = 512;
constexpr int MAX_PROBLEMS = 3;

struct Problem {
  int M, N, bn;
  int nt, tiles;      // column tiles; tiles to compute
  int kchunks, passes;
  int a_mn, b_mn;
  int upper;          // M == N: only tiles that reach the diagonal or lie above it, in 128 x 128 blocks
  uint32_t idesc;
  void* D;            // M x N, pitch ldd: bf16 (out_mode 0) or fp32 (1: store, 2: add into), or
  void* D2;           // out_mode 3: D the hi and D2 the lo bf16 plane
  int64_t ldd;
  int out_mode;
  float alpha;
  const bf16* add;    // optional addend: D[i][j] += add[i * ldadd + j] (out_mode 0 or 3)
  int64_t ldadd;
  int tri, k0, k1;    // out_mode 4: which terms of the contraction can be other than zero
  int wide;           // every base and pitch of D, D2 and add is a multiple of 32 bytes
  // which pair computes which tile: tiles [0, lo_tiles) are dealt in turn to the lo_n pairs from
  // lo_first on (those with less work so far), the rest to all pairs in turn from rr0 on
  int lo_first, lo_n, lo_tiles, rr0;
};

struct GroupArgs {
  Problem p[MAX_PROBLEMS];
  int n;
  int* status;
  uint64_t timeout_ns;
};

struct GroupMaps {
  CUtensorMap a[MAX_PROBLEMS][2], b[MAX_PROBLEMS][2];  // first and second K pass
};

// Shared-memory descriptor of an MN-major operand tile written by TMA as 64-element (128-byte)
// swizzled rows, one row per K index: 8-row groups 1024 bytes apart along K (stride byte offset),
// 64-element MN blocks MN_BOX bytes apart (leading byte offset).
__device__ __forceinline__ uint64_t sw128_mn_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((MN_BOX >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Terms of element (i, j) over the contraction's columns [k0, k1) (triangular operands: GemmF64::tri).
__device__ __forceinline__ int terms(const Problem& q, int i, int j) {
  int a = q.k0, b = q.k1;
  if (q.tri & 1) a = max(a, j);
  if (q.tri & 4) a = max(a, i);
  if (q.tri & 2) b = min(b, j + 1);
  return max(b - a, 0);
}

// One lane's up to 32 consecutive values of a row: whole 32-byte sectors when `wide`, else 16-byte
// pieces (pitches are multiples of 16 bytes and columns start at multiples of 32), single values at
// a ragged end. bf16 values in pairs, 16 words.
template <int WORDS>
__device__ __forceinline__ void store_words(uint32_t* p, bool wide, const uint32_t (&v)[WORDS]) {
  if (wide) {
#pragma unroll
    for (int i = 0; i < WORDS; i += 8) stg256(p + i, v + i);
  } else {
#pragma unroll
    for (int i = 0; i < WORDS; i += 4) *reinterpret_cast<uint4*>(p + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
  }
}
template <int WORDS>
__device__ __forceinline__ void load_words(const uint32_t* p, bool wide, uint32_t* v) {
  if (wide) {
#pragma unroll
    for (int i = 0; i < WORDS; i += 8) ldg256_cg(p + i, v + i);
  } else {
#pragma unroll
    for (int i = 0; i < WORDS; i += 4) {
      const uint4 x = __ldcg(reinterpret_cast<const uint4*>(p + i));
      v[i] = x.x;
      v[i + 1] = x.y;
      v[i + 2] = x.z;
      v[i + 3] = x.w;
    }
  }
}
__device__ __forceinline__ void store_f32(float* p, int nc, bool wide, const uint32_t (&v)[32]) {
  if (nc == 32) {
    store_words(reinterpret_cast<uint32_t*>(p), wide, v);
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < nc) p[j] = __uint_as_float(v[j]);
  }
}
__device__ __forceinline__ void load_f32(const float* p, int nc, bool wide, uint32_t (&v)[32]) {
  if (nc == 32) {
    load_words<32>(reinterpret_cast<const uint32_t*>(p), wide, v);
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = j < nc ? __float_as_uint(__ldcg(p + j)) : 0u;
  }
}
__device__ __forceinline__ void store_b16(bf16* p, int nc, bool wide, const uint32_t (&v)[16]) {
  if (nc == 32) {
    store_words(reinterpret_cast<uint32_t*>(p), wide, v);
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < nc) reinterpret_cast<uint16_t*>(p)[j] = (uint16_t)(v[j / 2] >> (16 * (j & 1)));
  }
}
__device__ __forceinline__ void load_b16(const bf16* p, int nc, bool wide, uint32_t (&v)[32]) {
  if (nc == 32) {
    load_words<16>(reinterpret_cast<const uint32_t*>(p), wide, v);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const unsigned short* s = reinterpret_cast<const unsigned short*>(p) + 2 * j;
      v[j] = (2 * j < nc ? (uint32_t)__ldcg(s) : 0u) | (2 * j + 1 < nc ? (uint32_t)__ldcg(s + 1) << 16 : 0u);
    }
  }
}

// The tiles of one pair, in order (the same for every role of both CTAs; m0 is this CTA's half).
struct TileIter {
  const GroupArgs& g;
  int p = 0, j = -1, phase = 0;
  int m0 = 0, n0 = 0;
  __device__ explicit TileIter(const GroupArgs& args) : g(args) {}
  __device__ void place(const Problem& q, int idx) {
    int mi, ni;
    if (q.upper) {  // row tile mi holds column tiles from mi 256 / bn on
      mi = 0;
      while (true) {
        const int first = mi * PM / q.bn, n = q.nt - first;
        if (idx < n) {
          ni = first + idx;
          break;
        }
        idx -= n;
        ++mi;
      }
    } else {
      mi = idx / q.nt;
      ni = idx % q.nt;
    }
    m0 = mi * PM + (int)(blockIdx.x & 1) * BM;
    n0 = ni * q.bn;
  }
  __device__ bool next() {
    const int G = (int)gridDim.x / 2, c = (int)blockIdx.x / 2;
    for (; p < g.n; ++p, phase = 0, j = -1) {
      const Problem& q = g.p[p];
      if (phase == 0) {
        if (j < 0) {
          const int lc = (c - q.lo_first + G) % G;
          j = lc < q.lo_n ? lc : q.lo_tiles;
        }
        if (j < q.lo_tiles) {
          place(q, j);
          j += q.lo_n;
          return true;
        }
        phase = 1;
        j = q.lo_tiles + (c - q.rr0 + G) % G;
      }
      if (j < q.tiles) {
        place(q, j);
        j += G;
        return true;
      }
    }
    return false;
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ GroupMaps maps, const __grid_constant__ GroupArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 2 * EPI_WARPS);  // the leader's: both CTAs' warps
    }
    mbar_init(drain, 1);
    fence_mbar_init();
    for (int i = 0; i < g.n; ++i)
      for (int k = 0; k < g.p[i].passes; ++k) {
        prefetch_tmap(&maps.a[i][k]);
        prefetch_tmap(&maps.b[i][k]);
      }
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are initialised before either signals the other's
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const bool leader = (blockIdx.x & 1) == 0;
  TileIter t(g);

  if (warp == 0 || warp == EPI_WARPS + 2) {
    if (lane == 0) {
      // ---------------- TMA producers: warp 0 loads A, the last warp B ----------------
      // (One thread issuing both, with the stage index by division and the boxes in a loop, was the
      // bound of MN-major products: 62 us of main loop where the MMAs take 34.)
      const bool is_a = warp == 0;
      pdl_wait_primary();
      int s = 0, it = 0;
      uint32_t ph = 1;  // parity that a fresh "empty" barrier passes
      bool dead = false;
      while (!dead && t.next()) {
        const Problem& q = g.p[t.p];
        const uint32_t bytes = 2 * A_BYTES + (uint32_t)q.bn * BK * 2;  // both CTAs' loads
        const bool mn = is_a ? q.a_mn : q.b_mn;
        const int hb = q.bn / 2, kch = q.kchunks;
        const int r0 = is_a ? t.m0 : t.n0 + (leader ? 0 : hb);
        const bool two = mn && (is_a || hb > 64);  // a second 64-wide MN-major box
        const uint32_t dst0 = smem_u32(smem) + (is_a ? 0u : A_BYTES);
        for (int pass = 0; pass < q.passes && !dead; ++pass) {
          const CUtensorMap* map = is_a ? &maps.a[t.p][pass] : &maps.b[t.p][pass];
          for (int k0 = 0; k0 < kch * BK; k0 += BK) {
            if (!mbar_wait(&empty[s], ph, g.timeout_ns)) {
              latch_status(g.status, PIFA_ERR_TIMEOUT);
              dead = true;
              break;
            }
            const uint32_t dst = dst0 + (uint32_t)s * STAGE_BYTES;
            const uint32_t bar = mapa_shared(smem_u32(&full[s]), 0);  // the leader's barrier counts both CTAs' bytes
            if (leader && is_a) mbar_arrive_expect_tx(&full[s], bytes);
            if (mn) {
              tma_load_2d_pair(dst, map, r0, k0, bar);
              if (two) tma_load_2d_pair(dst + MN_BOX, map, r0 + 64, k0, bar);
            } else {
              tma_load_2d_pair(dst, map, k0, r0, bar);
            }
            if (++s == STAGES) {
              s = 0;
              ph ^= 1u;
            }
            ++it;
          }
        }
      }
      if (dead) linger(100000000ull);
      // nothing may land in shared memory after the CTA has left: the leader waits for both CTAs'
      // copies, and the cluster barrier at the end holds the other CTA until it has
      for (int i = it > STAGES ? it - STAGES : 0; leader && is_a && i < it; ++i)
        if (!mbar_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u, 100000000ull))
          latch_status(g.status, PIFA_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ---------------- MMA issuer (the leader's, for both CTAs) ----------------
      int n = 0, s = 0;
      uint32_t ph = 0;
      bool dead = false;
      for (; !dead && t.next(); ++n) {
        const Problem& q = g.p[t.p];
        const int total = q.kchunks * q.passes, buf = n & 1;
        const uint32_t idesc = q.idesc, acc = tmem + (uint32_t)(buf * BNMAX);
        // K-major tiles advance 32 bytes along a swizzled row per K = 16; MN-major tiles advance 16
        // rows (2048 bytes); descriptors count 16-byte units
        const uint32_t base = smem_u32(smem);
        const uint64_t a0 = q.a_mn ? sw128_mn_desc(base) : sw128_desc(base);
        const uint64_t b0 = q.b_mn ? sw128_mn_desc(base + A_BYTES) : sw128_desc(base + A_BYTES);
        const uint32_t da = q.a_mn ? 128u : 2u, db = q.b_mn ? 128u : 2u;
        if (n >= 2 && !mbar_wait_cluster(&acce[buf], (uint32_t)((n >> 1) - 1) & 1u, g.timeout_ns)) {
          dead = true;
          break;
        }
        tc_fence_after();
        for (int i = 0; i < total; ++i) {
          if (!mbar_wait(&full[s], ph, g.timeout_ns)) {
            dead = true;
            break;
          }
          tc_fence_after();
          const uint32_t so = (uint32_t)s * (STAGE_BYTES / 16);
#pragma unroll
          for (uint32_t kk = 0; kk < BK / 16; ++kk)
            mma_bf16_ss_pair(acc, a0 + (so + kk * da), b0 + (so + kk * db), idesc, (i > 0 || kk > 0) ? 1u : 0u);
          mma_commit_pair(&empty[s]);
          if (++s == STAGES) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!dead) mma_commit_pair(&accf[buf]);
      }
      if (dead) latch_status(g.status, PIFA_ERR_TIMEOUT);
      mma_commit_pair(drain);  // every MMA has completed before the pair frees its tensor memory
      if (!mbar_wait(drain, 0, 100000000ull)) latch_status(g.status, PIFA_ERR_TIMEOUT);
    }
  } else {
    // ---------------- epilogue: warps 2..9, TMEM lane quarter warp % 4 ----------------
    // The two warps of a quarter take its 32-column blocks in turn. A lane holds 32 consecutive values
    // of one row of D and writes them straight from its registers as whole 32-byte sectors (16-byte
    // pieces where a base or pitch is no multiple of 32 bytes, single values at a ragged end). A
    // transpose through shared memory in front of 4-byte stores took about 9 us per tile.
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    for (int n = 0; t.next(); ++n) {
      const Problem& q = g.p[t.p];
      const int buf = n & 1;
      const int row = t.m0 + q4 * 32 + lane;
      const int ncols = min(q.bn, q.N - t.n0);
      const int mode = q.out_mode;
      const float alpha = q.alpha;
      if (!__all_sync(0xffffffffu, mbar_wait(&accf[buf], (uint32_t)(n >> 1) & 1u, g.timeout_ns))) {
        latch_status(g.status, PIFA_ERR_TIMEOUT);
        break;
      }
      tc_fence_after();
      for (int c0 = half * 32; c0 < ncols; c0 += 64) {
        const int col = t.n0 + c0;
        if (q.upper && (col & ~127) + BM <= t.m0) continue;  // a 128 x 128 block below the diagonal
        const int64_t o = (int64_t)row * q.ldd + col;
        const int nc = row < q.M ? min(32, q.N - col) : 0;  // columns this lane writes
        uint32_t v[32], old[32];
        if (mode == 2 && nc > 0)  // the values to add to, in flight while the accumulator is read
          load_f32(reinterpret_cast<const float*>(q.D) + o, nc, q.wide, old);
        if (q.add && nc > 0) load_b16(q.add + (int64_t)row * q.ldadd + col, nc, q.wide, old);
        __syncwarp();
        tmem_ld_32x32b_x32(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * BNMAX + c0), v);
        tmem_ld_wait();
        if (nc <= 0) continue;
        if (mode == 1 || mode == 2) {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            float f = __uint_as_float(v[j]) * alpha;
            if (mode == 2) f += __uint_as_float(old[j]);
            v[j] = __float_as_uint(f);
          }
          store_f32(reinterpret_cast<float*>(q.D) + o, nc, q.wide, v);
        } else if (mode == 4) {  // one word of 32 columns per lane
          uint32_t word = 0;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float f = __uint_as_float(v[j]);
            const bool low = f != 0.0f && !(f * f >= alpha * alpha * (float)terms(q, row, col + j));
            word |= (low && j < nc ? 1u : 0u) << j;
          }
          reinterpret_cast<uint32_t*>(q.D)[(int64_t)row * q.ldd + (col >> 5)] = word;
        } else {
          uint32_t h[16], l[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float f0 = __uint_as_float(v[2 * j]) * alpha, f1 = __uint_as_float(v[2 * j + 1]) * alpha;
            if (q.add) {
              f0 += __uint_as_float(old[j] << 16);
              f1 += __uint_as_float(old[j] & 0xffff0000u);
            }
            const __nv_bfloat162 hb = __floats2bfloat162_rn(f0, f1);
            const __nv_bfloat162 lb = __floats2bfloat162_rn(f0 - __low2float(hb), f1 - __high2float(hb));
            h[j] = *reinterpret_cast<const uint32_t*>(&hb);
            l[j] = *reinterpret_cast<const uint32_t*>(&lb);
          }
          store_b16(reinterpret_cast<bf16*>(q.D) + o, nc, q.wide, h);
          if (mode == 3) store_b16(reinterpret_cast<bf16*>(q.D2) + o, nc, q.wide, l);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(mapa_shared(smem_u32(&acce[buf]), 0));  // this warp has read its share
    }
  }

  // Every wait above is bounded, so every thread of both CTAs gets here: no CTA frees its tensor
  // memory or leaves while the pair's MMAs, copies or arrivals may still reach it.
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

// Pairs of CTAs that run at once on the current device: two SMs each, as many as its SM groups give. A query
// that fails counts as one for this call and is made again by the next.
int pair_count() {
  static std::mutex mu;
  static std::map<int, int> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = known.find(dev);
  if (it != known.end()) return it->second;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int m = 0;
  if (dev < 0 || cudaOccupancyMaxActiveClusters(&m, gemm_tc_kernel, &cfg) != cudaSuccess || m < 1) {
    cudaGetLastError();  // leaves no sticky error behind
    return 1;
  }
  return known[dev] = m;
}

int tile_width(const GemmTc& g, int want) {
  const int64_t unit = g.b_mn ? 128 : 32;  // two halves, of 64-column boxes where B is MN-major
  const int64_t n = g.N >= want ? want : g.N;
  return (int)((n + unit - 1) / unit * unit);
}

int64_t tile_count(const GemmTc& g, int bn) {
  const int64_t mt = (g.M + PM - 1) / PM, nt = (g.N + bn - 1) / bn;
  if (!g.upper) return mt * nt;
  int64_t n = 0;
  for (int64_t i = 0; i < mt; ++i) n += nt - i * PM / bn;
  return n;
}

// Relative time of one tile: a 64-column K step costs about the bytes of its operands (the MMAs of
// a 256-wide tile take as long), and a tile's start and its share of the last epilogue about four.
int64_t tile_cost(const GemmTc& g, int bn) {
  return ((g.K + BK - 1) / BK * ((g.A2 || g.B2) ? 2 : 1) + 4) * (PM + bn);
}

}  // namespace

int gemm_tc_group(const GemmTc* gs, int n, int* status, uint64_t timeout_ns, cudaStream_t stream) {
  const int64_t lim = (int64_t)1 << 30;
  const GemmTc* order[MAX_PROBLEMS];
  int np = 0;
  for (int i = 0; i < n; ++i) {
    const GemmTc& g = gs[i];
    if (g.M <= 0 || g.N <= 0) continue;
    if (np == MAX_PROBLEMS) return pifa_fail(PIFA_ERR_INVALID_ARG, "gemm_tc: too many products");
    if (g.K <= 0) return pifa_fail(PIFA_ERR_INVALID_ARG, "gemm_tc: K must be positive");
    if (g.M >= lim || g.N >= lim || g.K >= lim) return pifa_fail(PIFA_ERR_INVALID_ARG, "gemm_tc: size >= 2^30");
    if (g.upper && g.M != g.N) return pifa_fail(PIFA_ERR_INVALID_ARG, "gemm_tc: upper triangle of a non-square product");
    if (g.add && g.out_mode != 0 && g.out_mode != 3)
      return pifa_fail(PIFA_ERR_UNSUPPORTED, "gemm_tc: addend of an fp32 product");
    order[np++] = &g;
  }
  if (np == 0) return PIFA_OK;
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e != cudaSuccess) return pifa_fail_cuda("cudaFuncSetAttribute(gemm_tc)", e);
  const int G = pair_count();  // pairs of CTAs

  // Tile width: the widest (256, 128, 64) whose most loaded pair finishes first; the same for
  // every product of the launch. The tiles of the costliest product are dealt first, and the next
  // ones fill up the pairs that got fewer.
  GroupArgs a = {};
  const GemmTc* slot[MAX_PROBLEMS] = {};
  int64_t best = -1;
  for (int want = BNMAX; want >= 64; want /= 2) {
    const GemmTc* o[MAX_PROBLEMS];
    for (int i = 0; i < np; ++i) {  // by falling cost of a tile
      int k = i;
      while (k > 0 && tile_cost(*o[k - 1], tile_width(*o[k - 1], want)) < tile_cost(*order[i], tile_width(*order[i], want))) {
        o[k] = o[k - 1];
        --k;
      }
      o[k] = order[i];
    }
    GroupArgs c = {};
    // CTAs [hs, hs + hn) (around the grid) carry `extra` more than the others, which carry `base`
    int64_t base = 0, extra = 0, hs = 0, hn = 0;
    bool fits = true;
    for (int i = 0; i < np; ++i) {
      const int bn = tile_width(*o[i], want);
      const int64_t tiles = tile_count(*o[i], bn), cost = tile_cost(*o[i], bn);
      if (tiles >= lim || (o[i]->N + bn - 1) / bn >= lim) fits = false;
      Problem& q = c.p[i];
      q.lo_first = (int)((hs + hn) % G);
      q.lo_n = (int)(G - hn);
      const int64_t fill = q.lo_n * (extra / cost);
      q.lo_tiles = (int)(tiles < fill ? tiles : fill);
      q.rr0 = q.lo_first;
      const int64_t rest = tiles - q.lo_tiles, rem = rest % G;
      const int64_t left = extra - (fill > 0 && q.lo_tiles == fill ? extra / cost * cost : 0);  // the low CTAs still lack this
      base += extra - left + rest / G * cost;
      extra = left;
      if (rem > 0) {  // the first `rem` CTAs from rr0 on, the low ones foremost, get one tile more
        hs = q.rr0;
        hn = rem;
        extra = rem > q.lo_n ? cost + left : (cost > left ? cost : left);
      }
    }
    const int64_t load = base + extra;
    if (!fits) continue;
    if (best < 0 || load < best) {
      best = load;
      for (int i = 0; i < np; ++i) {
        Problem& q = c.p[i];
        q.bn = tile_width(*o[i], want);
        q.tiles = (int)tile_count(*o[i], q.bn);
      }
      a = c;
      a.n = np;
      for (int i = 0; i < np; ++i) slot[i] = o[i];
    }
  }
  if (best < 0) return pifa_fail(PIFA_ERR_UNSUPPORTED, "gemm_tc: more than 2^30 tiles");

  GroupMaps maps = {};
  for (int i = 0; i < np; ++i) {
    const GemmTc& g = *slot[i];
    Problem& q = a.p[i];
    q.M = (int)g.M;
    q.N = (int)g.N;
    q.nt = (int)((g.N + q.bn - 1) / q.bn);
    q.kchunks = (int)((g.K + BK - 1) / BK);
    q.passes = (g.A2 || g.B2) ? 2 : 1;
    q.a_mn = g.a_mn;
    q.b_mn = g.b_mn;
    q.upper = g.upper;
    q.idesc = idesc_bf16_f32(PM, (uint32_t)q.bn) | (g.a_mn ? (1u << 15) : 0u) | (g.b_mn ? (1u << 16) : 0u);
    q.D = g.D;
    q.D2 = g.D2;
    q.ldd = g.ldd;
    q.out_mode = g.out_mode;
    q.alpha = g.alpha;
    q.add = reinterpret_cast<const bf16*>(g.add);
    q.ldadd = g.ldadd;
    q.tri = g.tri;
    q.k0 = g.k0;
    q.k1 = g.k1;
    const int64_t esz = (g.out_mode == 1 || g.out_mode == 2) ? 4 : 2;
    q.wide = ((reinterpret_cast<uintptr_t>(g.D) | reinterpret_cast<uintptr_t>(g.D2) | (uintptr_t)(g.ldd * esz) |
               reinterpret_cast<uintptr_t>(g.add) | (uintptr_t)(g.add ? g.ldadd * 2 : 0)) & 31u) == 0;
    int st;
    for (int k = 0; k < 2; ++k) {
      const void* A = k && g.A2 ? g.A2 : g.A;
      const void* B = k && g.B2 ? g.B2 : g.B;
      if ((st = g.a_mn ? make_tmap_2d(&maps.a[i][k], PIFA_DTYPE_BF16, A, g.K, g.M, g.lda, 64, BK)
                       : make_tmap_2d(&maps.a[i][k], PIFA_DTYPE_BF16, A, g.M, g.K, g.lda, BK, BM)) != PIFA_OK)
        return st;
      if ((st = g.b_mn ? make_tmap_2d(&maps.b[i][k], PIFA_DTYPE_BF16, B, g.K, g.N, g.ldb, 64, BK)
                       : make_tmap_2d(&maps.b[i][k], PIFA_DTYPE_BF16, B, g.N, g.K, g.ldb, BK, (uint32_t)q.bn / 2)) != PIFA_OK)
        return st;
    }
  }
  a.status = status;
  a.timeout_ns = timeout_ns;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (unsigned)G);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  e = pifa_launch_ex(&cfg, gemm_tc_kernel, maps, a);
  if (e != cudaSuccess) return pifa_fail_cuda("gemm_tc launch", e);
  return PIFA_OK;
}
