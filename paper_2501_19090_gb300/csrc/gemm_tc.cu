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
//   B2 in place of B (same layouts) consumes such a pair: D = (A + A2) B^T or A (B + B2)^T.
//
// One launch computes up to three independent products. The grid is persistent, one CTA of 320
// threads per SM: warp 0 issues TMA loads into a 4-stage ring that runs on from tile to tile, warp 1
// issues tcgen05.mma (M = 128, N = bn <= 256, K = 16) from one thread into one of two accumulators
// (256 TMEM columns each), and warps 2-9 drain the other one meanwhile, so that the conversions,
// the values to add in and the stores of a tile run under the next tile's MMAs. What this replaced,
// one launch per product of one CTA per tile (two CTAs per SM of 128-wide tiles, or one of 256-wide
// ones with a third of its time in the epilogue, products on side streams), kept the tensor cores
// 27-45% busy. 4096 x 4096, r = 2048, T = 2048: backward 317.1 -> 253.6 us, the M accumulators of
// two batches 860.8 -> 538.1 us, every output bit for bit the same.
// Every wait is bounded (globaltimer); on timeout the CTA latches PIFA_ERR_TIMEOUT, drains what it
// has in flight and returns.
#include <cuda_bf16.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"

namespace {

using namespace pifa;
using bf16 = __nv_bfloat16;

constexpr int BM = 128;
constexpr int BNMAX = 256;
constexpr int BK = 64;
constexpr int STAGES = 4;
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 64 + 32 * EPI_WARPS;
constexpr uint32_t A_BYTES = BM * BK * 2;             // 16 KB
constexpr uint32_t STAGE_BYTES = A_BYTES + BNMAX * BK * 2;
constexpr uint32_t MN_BOX = 64 * BK * 2;              // one MN-major box: 64 (MN) x 64 (K), 8 KB
constexpr uint32_t TILE_FLOATS = 32 * 33;             // an epilogue warp's transpose tile
constexpr size_t SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + EPI_WARPS * TILE_FLOATS * 4 + 256;
constexpr uint32_t TMEM_COLS = 512;
constexpr int MAX_PROBLEMS = 3;

struct Problem {
  int M, N, bn;
  int mt, nt, tiles;  // row tiles, column tiles, tiles to compute
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
  // which CTA computes which tile: tiles [0, lo_tiles) are dealt in turn to the lo_n CTAs from
  // lo_first on (those with less work so far), the rest to all CTAs in turn from rr0 on
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

// The tiles of one CTA, in order (the same for every role of the CTA).
struct TileIter {
  const GroupArgs& g;
  int p = 0, j = -1, phase = 0;
  int m0 = 0, n0 = 0;
  __device__ explicit TileIter(const GroupArgs& args) : g(args) {}
  __device__ void place(const Problem& q, int idx) {
    int mi, ni;
    if (q.upper) {  // row tile mi holds column tiles from mi 128 / bn on
      mi = 0;
      while (true) {
        const int first = mi * BM / q.bn, n = q.nt - first;
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
    m0 = mi * BM;
    n0 = ni * q.bn;
  }
  __device__ bool next() {
    const int G = (int)gridDim.x, c = (int)blockIdx.x;
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

__global__ void __launch_bounds__(THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ GroupMaps maps, const __grid_constant__ GroupArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* tiles_sm = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles_sm + EPI_WARPS * TILE_FLOATS);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], EPI_WARPS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    for (int i = 0; i < g.n; ++i)
      for (int k = 0; k < g.p[i].passes; ++k) {
        prefetch_tmap(&maps.a[i][k]);
        prefetch_tmap(&maps.b[i][k]);
      }
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  TileIter t(g);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      pdl_wait_primary();
      int it = 0;
      bool dead = false;
      while (!dead && t.next()) {
        const Problem& q = g.p[t.p];
        const uint32_t bytes = A_BYTES + (uint32_t)q.bn * BK * 2;
        const bool amn = q.a_mn, bmn = q.b_mn;
        const int nb = q.bn / 64, kch = q.kchunks, m0 = t.m0, n0 = t.n0;
        for (int pass = 0; pass < q.passes && !dead; ++pass) {
          const CUtensorMap* ma = &maps.a[t.p][pass];
          const CUtensorMap* mb = &maps.b[t.p][pass];
          for (int kc = 0; kc < kch; ++kc, ++it) {
            const int s = it % STAGES;
            if ((it >= STAGES && !mbar_wait(&empty[s], (uint32_t)((it / STAGES) - 1) & 1u, g.timeout_ns)) || *abort_flag) {
              latch_status(g.status, PIFA_ERR_TIMEOUT);
              *abort_flag = 1;
              dead = true;
              break;
            }
            const uint32_t sa = smem_u32(smem + s * STAGE_BYTES), sb = sa + A_BYTES;
            const int k0 = kc * BK;
            mbar_arrive_expect_tx(&full[s], bytes);
            if (amn) {
              tma_load_2d(sa, ma, m0, k0, &full[s]);
              tma_load_2d(sa + MN_BOX, ma, m0 + 64, k0, &full[s]);
            } else {
              tma_load_2d(sa, ma, k0, m0, &full[s]);
            }
            if (bmn) {
              for (int h = 0; h < nb; ++h) tma_load_2d(sb + h * MN_BOX, mb, n0 + 64 * h, k0, &full[s]);
            } else {
              tma_load_2d(sb, mb, k0, n0, &full[s]);
            }
          }
        }
      }
      // nothing may land in shared memory after the CTA has left
      for (int i = it > STAGES ? it - STAGES : 0; i < it; ++i)
        if (!mbar_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u, 100000000ull))
          latch_status(g.status, PIFA_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      int it = 0, n = 0;
      bool dead = false;
      for (; !dead && t.next(); ++n) {
        const Problem& q = g.p[t.p];
        const int total = q.kchunks * q.passes, buf = n & 1;
        const uint32_t idesc = q.idesc, acc = tmem + (uint32_t)(buf * BNMAX);
        const bool amn = q.a_mn, bmn = q.b_mn;
        if (n >= 2 && !mbar_wait(&acce[buf], (uint32_t)((n >> 1) - 1) & 1u, g.timeout_ns)) {
          dead = true;
          break;
        }
        tc_fence_after();
        for (int i = 0; i < total; ++i, ++it) {
          const int s = it % STAGES;
          if (!mbar_wait(&full[s], (uint32_t)(it / STAGES) & 1u, g.timeout_ns) || *abort_flag) {
            dead = true;
            break;
          }
          tc_fence_after();
          const uint32_t a = smem_u32(smem + s * STAGE_BYTES), b = a + A_BYTES;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            // K-major tiles advance 32 bytes along a swizzled row per K = 16; MN-major tiles advance
            // 16 rows (2048 bytes)
            const uint64_t ad = amn ? sw128_mn_desc(a + kk * 2048) : sw128_desc(a + kk * 32);
            const uint64_t bd = bmn ? sw128_mn_desc(b + kk * 2048) : sw128_desc(b + kk * 32);
            mma_bf16_ss(acc, ad, bd, idesc, (i > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit(&empty[s]);
        }
        if (!dead) mma_commit(&accf[buf]);
      }
      if (dead) {
        latch_status(g.status, PIFA_ERR_TIMEOUT);
        *abort_flag = 1;
      }
      mma_commit(drain);  // every MMA has completed before the CTA frees its tensor memory
      if (!mbar_wait(drain, 0, 100000000ull)) latch_status(g.status, PIFA_ERR_TIMEOUT);
    }
  } else {
    // ---------------- epilogue: warps 2..9, TMEM lane quarter warp % 4 ----------------
    // The two warps of a quarter take its 32-column blocks in turn. A block (32 rows, 32 columns) is
    // read from TMEM one row per lane and goes through this warp's shared-memory tile, so that a
    // store instruction covers consecutive columns (one row of fp32, two rows of bf16 pairs).
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    float* tile = tiles_sm + (warp - 2) * TILE_FLOATS;
    for (int n = 0; t.next(); ++n) {
      const Problem& q = g.p[t.p];
      const int buf = n & 1;
      const int r0 = t.m0 + q4 * 32, nrows = min(32, q.M - r0);
      const int ncols = min(q.bn, q.N - t.n0);
      const int mode = q.out_mode;
      bool ok = mbar_wait(&accf[buf], (uint32_t)(n >> 1) & 1u, g.timeout_ns) && !*abort_flag;
      if (!__all_sync(0xffffffffu, ok)) {
        latch_status(g.status, PIFA_ERR_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      tc_fence_after();
      for (int c0 = half * 32; c0 < ncols; c0 += 64) {
        const int col0 = t.n0 + c0;
        if (q.upper && (col0 & ~127) + BM <= t.m0) continue;  // a 128 x 128 block below the diagonal
        float old[32];
        if (mode == 2) {  // the values to add to, in flight while the accumulator is read
          const float* d = reinterpret_cast<const float*>(q.D) + (int64_t)r0 * q.ldd + col0 + lane;
#pragma unroll
          for (int rr = 0; rr < 32; ++rr)
            old[rr] = (rr < nrows && col0 + lane < q.N) ? __ldcg(d + (int64_t)rr * q.ldd) : 0.0f;
        }
        uint32_t v[32];
        tmem_ld_32x32b_x32(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * BNMAX + c0), v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) tile[lane * 33 + j] = __uint_as_float(v[j]) * q.alpha;
        __syncwarp();
        if (mode == 1 || mode == 2) {
          float* d = reinterpret_cast<float*>(q.D) + (int64_t)r0 * q.ldd + col0 + lane;
          if (col0 + lane < q.N) {
#pragma unroll
            for (int rr = 0; rr < 32; ++rr)
              if (rr < nrows) d[(int64_t)rr * q.ldd] = mode == 2 ? tile[rr * 33 + lane] + old[rr] : tile[rr * 33 + lane];
          }
        } else {
          // two rows per step, a pair of columns per lane (col is even and the pitches are multiples
          // of 8: 4-byte aligned)
          const int rl = lane >> 4, cl = (lane & 15) * 2, col = col0 + cl;
          const bool two = col + 1 < q.N, in = col < q.N;
          uint32_t av[16];
          if (q.add) {
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const bf16* s = q.add + (int64_t)(r0 + 2 * u + rl) * q.ldadd + col;
              av[u] = 0u;
              if (2 * u + rl < nrows && in)
                av[u] = two ? __ldcg(reinterpret_cast<const unsigned int*>(s))
                            : (uint32_t)__ldcg(reinterpret_cast<const unsigned short*>(s));
            }
          }
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int rr = 2 * u + rl;
            if (rr >= nrows || !in) continue;
            float f0 = tile[rr * 33 + cl], f1 = tile[rr * 33 + cl + 1];
            if (q.add) {
              f0 += __uint_as_float(av[u] << 16);
              f1 += __uint_as_float(av[u] & 0xffff0000u);
            }
            const int64_t o = (int64_t)(r0 + rr) * q.ldd + col;
            const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
            bf16* d = reinterpret_cast<bf16*>(q.D) + o;
            if (two) *reinterpret_cast<__nv_bfloat162*>(d) = h;
            else *d = h.x;
            if (mode == 3) {
              const __nv_bfloat162 l = __floats2bfloat162_rn(f0 - __low2float(h), f1 - __high2float(h));
              bf16* d2 = reinterpret_cast<bf16*>(q.D2) + o;
              if (two) *reinterpret_cast<__nv_bfloat162*>(d2) = l;
              else *d2 = l.x;
            }
          }
        }
        __syncwarp();  // the next block reuses the tile
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[buf]);  // this warp has read its share of the accumulator
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

int sm_count_gemm() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      n = 1;
  }
  return n;
}

int tile_width(const GemmTc& g, int want) {
  const int64_t unit = g.b_mn ? 64 : 16;  // MN-major B tiles come in 64-column boxes
  return (int)(g.N >= want ? want : (g.N + unit - 1) / unit * unit);
}

int64_t tile_count(const GemmTc& g, int bn) {
  const int64_t mt = (g.M + BM - 1) / BM, nt = (g.N + bn - 1) / bn;
  if (!g.upper) return mt * nt;
  int64_t n = 0;
  for (int64_t i = 0; i < mt; ++i) n += nt - i * BM / bn;
  return n;
}

// Relative time of one tile: a 64-column K step costs about the bytes of its operands (the MMAs of
// a 256-wide tile take as long), and a tile's start and its share of the last epilogue about four.
int64_t tile_cost(const GemmTc& g, int bn) {
  return ((g.K + BK - 1) / BK * ((g.A2 || g.B2) ? 2 : 1) + 4) * (BM + bn);
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
    if (g.add && (g.out_mode == 1 || g.out_mode == 2))
      return pifa_fail(PIFA_ERR_UNSUPPORTED, "gemm_tc: addend of an fp32 product");
    order[np++] = &g;
  }
  if (np == 0) return PIFA_OK;
  const int G = sm_count_gemm();

  // Tile width: the widest (256, 192, 128, 64) whose most loaded CTA finishes first; the same for
  // every product of the launch. The tiles of the costliest product are dealt first, and the next
  // ones fill up the CTAs that got fewer.
  GroupArgs a = {};
  const GemmTc* slot[MAX_PROBLEMS] = {};
  int64_t best = -1;
  for (int want = BNMAX; want >= 64; want -= 64) {
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
    q.mt = (int)((g.M + BM - 1) / BM);
    q.nt = (int)((g.N + q.bn - 1) / q.bn);
    q.kchunks = (int)((g.K + BK - 1) / BK);
    q.passes = (g.A2 || g.B2) ? 2 : 1;
    q.a_mn = g.a_mn;
    q.b_mn = g.b_mn;
    q.upper = g.upper;
    q.idesc = idesc_bf16_f32(BM, (uint32_t)q.bn) | (g.a_mn ? (1u << 15) : 0u) | (g.b_mn ? (1u << 16) : 0u);
    q.D = g.D;
    q.D2 = g.D2;
    q.ldd = g.ldd;
    q.out_mode = g.out_mode;
    q.alpha = g.alpha;
    q.add = reinterpret_cast<const bf16*>(g.add);
    q.ldadd = g.ldadd;
    int st;
    for (int k = 0; k < 2; ++k) {
      const void* A = k && g.A2 ? g.A2 : g.A;
      const void* B = k && g.B2 ? g.B2 : g.B;
      if ((st = g.a_mn ? make_tmap_2d(&maps.a[i][k], PIFA_DTYPE_BF16, A, g.K, g.M, g.lda, 64, BK)
                       : make_tmap_2d(&maps.a[i][k], PIFA_DTYPE_BF16, A, g.M, g.K, g.lda, BK, BM)) != PIFA_OK)
        return st;
      if ((st = g.b_mn ? make_tmap_2d(&maps.b[i][k], PIFA_DTYPE_BF16, B, g.K, g.N, g.ldb, 64, BK)
                       : make_tmap_2d(&maps.b[i][k], PIFA_DTYPE_BF16, B, g.N, g.K, g.ldb, BK, (uint32_t)q.bn)) != PIFA_OK)
        return st;
    }
  }
  a.status = status;
  a.timeout_ns = timeout_ns;
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e != cudaSuccess) return pifa_fail_cuda("cudaFuncSetAttribute(gemm_tc)", e);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)G);
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
