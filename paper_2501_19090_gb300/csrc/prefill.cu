// prefill.cu -- PIFA forward for many tokens on the 5th-generation tensor cores (tcgen05).
//
// Split variant: two launches of one warp-specialised tcgen05 GEMM.
//   GEMM 1 (Algorithm 2, steps 2 and 4): D1 = W_p X^T, weight rows x tokens.
//           Epilogue writes bf16(Y_p) into the pivot columns Y[:, I[j]] and the pair
//           hi = rnd(Y_p), lo = rnd(Y_p - hi) into two T x r scratch matrices, rnd rounding to
//           C's storage type (bf16 or fp16).
//   GEMM 2 (Algorithm 2, steps 3 and 5): D2 = C [hi | lo]^T accumulated over K = r twice (hi pass
//           then lo pass), epilogue writes bf16(Y_np) into Y[:, I^c[i]].
// Weight rows are the MMA M dimension and tokens the N dimension, so the accumulator in tensor
// memory holds one weight row per TMEM lane: an epilogue warp's 32 lanes are 32 consecutive
// weight rows, which for a fixed token land in 32 ascending output columns of one row of Y.
//
// A pair of CTAs (one per SM, 352 threads each) computes a tile of 256 weight rows x bn tokens
// (bn <= 256) with pair MMAs (cta_group::2: M = 256, N = bn, K = 16): each CTA loads its 128 weight
// rows and half of the tile's tokens per 64 columns of K into a ring of stages (128-byte swizzle),
// warp 0 the weights, which need not wait for the previous kernel, the last warp the activations;
// the even CTA's warp 1 issues the MMAs of both; warps 2-9 of each CTA drain its 128 rows of the
// accumulator through tcgen05.ld. The grid is persistent with two accumulators (256 TMEM columns
// each), so that from the second tile on a tile's epilogue runs under the next tile's MMAs.
// Y's stores are a column scatter of 2 bytes per lane; Y_p's hi/lo planes go out as 4-byte stores of
// two rows after an exchange between neighbouring lanes. Every wait is bounded (globaltimer); on timeout the CTA
// latches PIFA_ERR_TIMEOUT, drains what it has in flight and returns.
//
// A 64-column chunk of K costs a tile 330 + 0.85 bn cycles by a pair (its MMAs are 2 bn of them) and
// 410 + 0.3 bn to 480 + 0.66 bn by one CTA, much of it the hand-offs of a stage (its copy's arrival, the
// MMAs' issue and commit, the release), which is why a stage holds two chunks where the ring allows, why
// the issuing threads do no division and read no flag, and why wide tiles are best where they fill
// the GPU. GEMMs of few tiles run on tiles of 128 rows by one CTA and split K: the 2 or 4 CTAs of a
// tile form a cluster, each accumulates its K-slice, stores the fp32 partial tile in its own freed
// ring, and the cluster adds the slices through distributed shared memory in a fixed order before the
// epilogue. pick_shape takes the form, width and split that these costs say finishes first. Measured beside
// every alternative in 398 GEMMs (20 layers, T = 80 to 4096), the call was 0.9% behind the best pick in the
// mean, more than 2% in 58 of them; the worst were layers whose rank is no multiple of 64 (4096 x 4096, r = 1638,
// T = 2048: 18%, one CTA where a pair's tiles would be read half as often).
// Against the one-CTA forms that this replaced (us, CUDA graph, one process): 7B attention T = 128
// 25.2 -> 20.0, 512 37.4 -> 34.6, 2048 58.0 -> 53.9, 4096 119.5 -> 94.7; 7B gate T = 2048 143.8 ->
// 120.4; 7B down T = 300 48.1 -> 35.9; 70B q/o T = 300 89.4 -> 56.3, 4096 400.3 -> 345.8; 70B gate/up
// T = 512 227.2 -> 181.5, 4096 1460.2 -> 1226.3. At T = 2048 on the 7B attention layer each GEMM is one
// round of 64 pair tiles: what is left is its 34 GFLOP at the tensor rate of 128 of 152 SMs (19 us), its
// launch and first copies (about 5 us) and its exposed epilogue (about 3 us).
#include <map>
#include <mutex>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "pifa.h"
#include "pifa_internal.h"
#include "ptx.cuh"

namespace {

using namespace pifa;
using bf16 = __nv_bfloat16;

constexpr int BM = 128;       // weight rows of one CTA
constexpr int PM = 2 * BM;    // of a pair
constexpr int BNMAX = 256;    // tokens per tile
constexpr int BK = 64;        // K per chunk: one 128-byte swizzle row of bf16
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 96 + 32 * EPI_WARPS;
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t RING_BYTES = 224 * 1024;
constexpr int MAX_STAGES = 10;
constexpr size_t SMEM_BYTES = 1024 + RING_BYTES + 256;
constexpr uint32_t TMEM_COLS = 512;

// Epilogue modes: what GEMM 1 also writes besides Y (GEMM 2 writes Y only).
enum { EPI_Y_ONLY = 0, EPI_SPLIT_BF16 = 1, EPI_SPLIT_F16 = 2 };

struct GemmArgs {
  uint32_t idesc;        // tcgen05 instruction descriptor (bf16 or fp16 operands)
  int M;                 // weight rows (r for GEMM 1, m - r for GEMM 2, times the groups)
  int N;                 // tokens T
  int bn;                // tokens per tile (MMA N): a multiple of 32, <= BNMAX
  int nt, mt, tiles;     // token tiles, row tiles
  int tok_fast;          // 1: consecutive tiles walk the token tiles (pairs of one weight-row block together)
  int gsz, mtg;          // weight rows per group (M when not grouped), row tiles per group: none spans two
  int goff;              // B columns between consecutive groups' K ranges (r; 0 when not grouped)
  int kchunks;           // ceil(K / 64) per pass
  int subs, ksteps;      // chunks per stage (1 or 2), stages per pass
  int passes;            // 1, or 2 for the hi + lo passes of GEMM 2
  int stages;
  uint32_t stage_bytes;
  const int32_t* cols;   // output column of each weight row (I or I^c)
  int m;                 // columns of Y (index bound)
  bf16* Y;
  int64_t ldy;
  void* yp_hi;           // GEMM 1 only: T x ldyp scratch, hi part (bf16 or fp16)
  void* yp_lo;           // lo part
  int64_t ldyp;
  int* status;
  uint64_t timeout_ns;
  int ks;                // K-slices per tile (kCl): CTAs of a cluster
};

// hi + lo split of an fp32 value in bf16 or fp16; fp16 saturates at +-65504 and reports it.
template <int kEpi>
__device__ __forceinline__ void split_hl(float f, uint16_t& h, uint16_t& l, bool& range_err) {
  if (kEpi == EPI_SPLIT_F16) {
    if (fabsf(f) > 65504.0f) {
      range_err = true;
      f = copysignf(65504.0f, f);
    }
    const __half hh = __float2half_rn(f);
    h = __half_as_ushort(hh);
    l = __half_as_ushort(__float2half_rn(f - __half2float(hh)));
  } else {
    const bf16 hh = __float2bfloat16_rn(f);
    h = __bfloat16_as_ushort(hh);
    l = __bfloat16_as_ushort(__float2bfloat16_rn(f - __bfloat162float(hh)));
  }
}

// kPair: a tile of 256 weight rows by a pair of CTAs; else of 128 rows by one.
// kCl (one-CTA tiles): split-K over a cluster of ks CTAs per tile (grids with too few tiles to fill the
// GPU): CTA z accumulates the K-steps [z total / ks, (z + 1) total / ks) of both passes; after a cluster
// barrier it adds rows [z 128 / ks, (z + 1) 128 / ks) of the slices in a fixed order.
template <int kEpi, bool kCl, bool kPair>
__global__ void __launch_bounds__(THREADS, 1)
    pifa_umma_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB0,
                   const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ GemmArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + RING_BYTES);
  uint64_t* empty = full + MAX_STAGES;
  uint64_t* accf = empty + MAX_STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  pdl_launch_dependents();  // the next kernel may launch now (its CTAs take SMs this grid leaves idle)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  static_assert(!(kCl && kPair), "split-K clusters are of one-CTA tiles");
  const bool leader = !kPair || (blockIdx.x & 1) == 0;  // issues the MMAs
  const int z = kCl ? (int)cluster_ctarank() : 0;
  const int ksteps = p.ksteps * p.passes;
  const int i0 = kCl ? (int)(((int64_t)z * ksteps) / p.ks) : 0;  // this CTA's K-steps [i0, i0 + total)
  const int total = kCl ? (int)(((int64_t)(z + 1) * ksteps) / p.ks) - i0 : ksteps;
  // tiles first, first + stride, ... of this CTA or pair
  const int first = kCl ? (int)blockIdx.x / p.ks : (int)blockIdx.x >> (kPair ? 1 : 0);
  const int stride = kCl ? p.tiles : (int)gridDim.x >> (kPair ? 1 : 0);
  auto place = [&](int idx, int& m0, int& mend, int& n0, int& bx0) {
    const int mi = p.tok_fast ? idx / p.nt : idx % p.mt, ni = p.tok_fast ? idx % p.nt : idx / p.mt;
    const int g = mi / p.mtg;
    m0 = g * p.gsz + (mi - g * p.mtg) * (kPair ? PM : BM) + (leader ? 0 : BM);  // this CTA's rows
    mend = min(p.M, (g + 1) * p.gsz);
    n0 = ni * p.bn;
    bx0 = g * p.goff;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], (kPair ? 2 : 1) * EPI_WARPS);  // the leader's: both CTAs' warps
    }
    mbar_init(drain, 1);
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB0);
    if (p.passes > 1) prefetch_tmap(&tmB1);
  }
  if (warp == 1) {
    if (kPair) {
      tmem_alloc_pair(tmem_slot, TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (kPair) cluster_sync_all();  // both CTAs' barriers are initialised before either signals the other's
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 || warp == EPI_WARPS + 2) {
    if (lane == 0) {
      // ---------------- TMA producers: warp 0 the weights, the last warp the activations ----------------
      const bool is_a = warp == 0;
      if (!is_a) pdl_wait_primary();  // X, or the y_p planes GEMM 1 wrote; the weights depend on no kernel
      const int hb = kPair ? p.bn / 2 : p.bn;  // this CTA's tokens
      const uint32_t bytes = (kPair ? 2 : 1) * A_BYTES + (uint32_t)p.bn * BK * 2;  // a chunk's, both CTAs'
      const uint32_t box = is_a ? A_BYTES : (uint32_t)hb * BK * 2;
      const uint32_t dst0 = smem_u32(smem) + (is_a ? 0u : (uint32_t)p.subs * A_BYTES);
      int s = 0, it = 0;
      uint32_t ph = 1;  // parity that a fresh "empty" barrier passes
      bool dead = false;
      for (int idx = first; idx < p.tiles && !dead; idx += stride) {
        int m0, mend, n0, bx0;
        place(idx, m0, mend, n0, bx0);
        const int y = is_a ? m0 : n0 + (leader ? 0 : hb), x0 = is_a ? 0 : bx0;
        const int pass = i0 / p.ksteps;
        int kc = (i0 - pass * p.ksteps) * p.subs;  // first chunk of the stage
        const CUtensorMap* map = is_a ? &tmA : pass ? &tmB1 : &tmB0;
        for (int i = 0; i < total; ++i, ++it) {
          if (!mbar_wait(&empty[s], ph, p.timeout_ns)) {
            latch_status(p.status, PIFA_ERR_TIMEOUT);
            dead = true;
            break;
          }
          const bool two = p.subs == 2 && kc + 1 < p.kchunks;
          if (leader && is_a) mbar_arrive_expect_tx(&full[s], two ? 2 * bytes : bytes);
          const uint32_t dst = dst0 + (uint32_t)s * p.stage_bytes;
          const int x = x0 + kc * BK;
          if (kPair) {
            const uint32_t bar = mapa_shared(smem_u32(&full[s]), 0);
            tma_load_2d_pair(dst, map, x, y, bar);
            if (two) tma_load_2d_pair(dst + box, map, x + BK, y, bar);
          } else {
            tma_load_2d(dst, map, x, y, &full[s]);
            if (two) tma_load_2d(dst + box, map, x + BK, y, &full[s]);
          }
          kc += p.subs;
          if (kc >= p.kchunks) {
            kc = 0;
            if (!is_a) map = &tmB1;
          }
          if (++s == p.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (dead) linger(100000000ull);
      // nothing may land in shared memory after the CTA has left: the leader waits for both CTAs'
      // copies, and the cluster barrier at the end holds the other CTA until it has
      for (int i = it > p.stages ? it - p.stages : 0; leader && is_a && i < it; ++i)
        if (!mbar_wait(&full[i % p.stages], (uint32_t)(i / p.stages) & 1u, 100000000ull))
          latch_status(p.status, PIFA_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ---------------- MMA issuer (the leader's, for both CTAs) ----------------
      int n = 0, s = 0;
      uint32_t ph = 0;
      bool dead = false;
      // descriptors count 16-byte units
      const uint64_t a0 = sw128_desc(smem_u32(smem)), b0 = sw128_desc(smem_u32(smem) + (uint32_t)p.subs * A_BYTES);
      const uint32_t step = p.stage_bytes / 16, boxb = (uint32_t)(kPair ? p.bn / 2 : p.bn) * 8u;
      auto commit = [](uint64_t* bar) {
        if (kPair) mma_commit_pair(bar);
        else mma_commit(bar);
      };
      for (int idx = first; idx < p.tiles && !dead; idx += stride, ++n) {
        const int buf = n & 1;
        const uint32_t acc = tmem + (uint32_t)(buf * BNMAX);
        const uint32_t pe = (uint32_t)((n >> 1) - 1) & 1u;
        if (n >= 2 && !(kPair ? mbar_wait_cluster(&acce[buf], pe, p.timeout_ns) : mbar_wait(&acce[buf], pe, p.timeout_ns))) {
          dead = true;
          break;
        }
        tc_fence_after();
        int kc = (i0 % p.ksteps) * p.subs;
        for (int i = 0; i < total; ++i) {
          if (!mbar_wait(&full[s], ph, p.timeout_ns)) {
            dead = true;
            break;
          }
          tc_fence_after();
          uint64_t a = a0 + (uint32_t)s * step, b = b0 + (uint32_t)s * step;
          const int n64 = p.subs == 2 && kc + 1 < p.kchunks ? 2 : 1;
          for (int u = 0; u < n64; ++u, a += A_BYTES / 16, b += boxb) {
#pragma unroll
            for (uint32_t kk = 0; kk < BK / 16; ++kk) {
              const uint32_t on = (i > 0 || u > 0 || kk > 0) ? 1u : 0u;
              if (kPair) mma_bf16_ss_pair(acc, a + kk * 2u, b + kk * 2u, p.idesc, on);
              else mma_bf16_ss(acc, a + kk * 2u, b + kk * 2u, p.idesc, on);
            }
          }
          kc += p.subs;
          if (kc >= p.kchunks) kc = 0;
          commit(&empty[s]);
          if (++s == p.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!dead) commit(&accf[buf]);
      }
      if (dead) latch_status(p.status, PIFA_ERR_TIMEOUT);
      commit(drain);  // every MMA has completed before the tensor memory is freed
      if (!mbar_wait(drain, 0, 100000000ull)) latch_status(p.status, PIFA_ERR_TIMEOUT);
    }
  } else {
    // ---------------- epilogue: warps 2..9, TMEM lane quarter warp % 4 ----------------
    // Warp w may access TMEM lanes 32 (w % 4) .. + 31, one quarter of the CTA's weight rows; the two
    // warps of a quarter take the tile's blocks of 32 tokens in turn.
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    bool range_err = false;
    int n = 0;
    for (int idx = first; idx < p.tiles; idx += stride, ++n) {
      int m0, mend, n0, bx0;
      place(idx, m0, mend, n0, bx0);
      const int buf = n & 1, ntok = min(p.bn, p.N - n0);
      const int row = m0 + q4 * 32 + lane;
      int col = -1;
      if (!kCl && row < mend) {
        col = __ldg(p.cols + row);
        if ((unsigned)col >= (unsigned)p.m) {
          latch_status(p.status, PIFA_ERR_DEVICE_INDEX);
          col = -1;
        }
      }
      if (!__all_sync(0xffffffffu, mbar_wait(&accf[buf], (uint32_t)(n >> 1) & 1u, p.timeout_ns))) {
        latch_status(p.status, PIFA_ERR_TIMEOUT);
        break;
      }
      tc_fence_after();
      if (kCl) fence_proxy_async_smem();  // the ring's last operands were read by the MMAs (async proxy)
      for (int c0 = half * 32; c0 < ntok; c0 += 64) {
        uint32_t v[32];
        tmem_ld_32x32b_x32(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * BNMAX + c0), v);
        tmem_ld_wait();
        if (kCl) {
          // this K-slice's partial tile into the ring as [token][128 rows] fp32 (the lanes of a
          // warp on consecutive rows): the cluster adds the slices below
          float* red = reinterpret_cast<float*>(smem) + c0 * BM + q4 * 32 + lane;
#pragma unroll
          for (int j = 0; j < 32; ++j) red[j * BM] = __uint_as_float(v[j]);
          continue;
        }
        bf16* y = p.Y + (int64_t)(n0 + c0) * p.ldy + col;
        const int nj = ntok - c0;
        // planes: lanes l and l ^ 1 exchange halves, so that a 4-byte store holds two neighbouring rows
        // of one token (even lanes token j, odd lanes j + 1): 64 contiguous bytes per 16 lanes
        const bool odd = lane & 1;
        const int64_t po = (int64_t)(n0 + c0 + (odd ? 1 : 0)) * p.ldyp + (row & ~1);
        const bool pin = kEpi != EPI_Y_ONLY && (row & ~1) < p.ldyp;  // rows beyond M hold zeros (padding columns)
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float f0 = __uint_as_float(v[j]), f1 = __uint_as_float(v[j + 1]);
          if (col >= 0 && j < nj) y[(int64_t)j * p.ldy] = __float2bfloat16_rn(f0);
          if (col >= 0 && j + 1 < nj) y[(int64_t)(j + 1) * p.ldy] = __float2bfloat16_rn(f1);
          if (kEpi != EPI_Y_ONLY) {
            uint16_t h0, l0, h1, l1;
            split_hl<kEpi>(f0, h0, l0, range_err);
            split_hl<kEpi>(f1, h1, l1, range_err);
            const uint32_t h = (uint32_t)h0 | (uint32_t)h1 << 16, l = (uint32_t)l0 | (uint32_t)l1 << 16;
            const uint32_t xh = __shfl_xor_sync(0xffffffffu, h, 1), xl = __shfl_xor_sync(0xffffffffu, l, 1);
            if (pin && j + (odd ? 1 : 0) < nj) {
              const int64_t o = po + (int64_t)j * p.ldyp;
              *reinterpret_cast<uint32_t*>(reinterpret_cast<uint16_t*>(p.yp_hi) + o) =
                  odd ? __byte_perm(xh, h, 0x7632) : __byte_perm(h, xh, 0x5410);
              *reinterpret_cast<uint32_t*>(reinterpret_cast<uint16_t*>(p.yp_lo) + o) =
                  odd ? __byte_perm(xl, l, 0x7632) : __byte_perm(l, xl, 0x5410);
            }
          }
        }
      }
      if (kCl) break;  // one tile per cluster
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {  // this warp has read its share of the accumulator
        if (kPair) mbar_arrive_remote(mapa_shared(smem_u32(&acce[buf]), 0));
        else mbar_arrive(&acce[buf]);
      }
    }
    if (range_err) latch_status(p.status, PIFA_ERR_RANGE);
  }

  // Every wait above is bounded, so every thread of every CTA gets here: no CTA frees its tensor
  // memory or leaves while the pair's MMAs, copies or arrivals may still reach it, and with kCl every
  // CTA of the cluster has its partial tile in its own shared memory.
  tc_fence_before();
  __syncthreads();
  if (kPair || kCl) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if (kPair) tmem_dealloc_pair(tmem, TMEM_COLS);
    else tmem_dealloc(tmem, TMEM_COLS);
  }
  if (kCl) {
    // CTA z finishes rows [z rpc, (z + 1) rpc) of the tile for all its tokens: four rows of a token
    // per thread and step, every slice's loads in flight at once, added in a fixed order (from its
    // own on, so that the CTAs do not all read one peer at a time). A second barrier keeps each CTA resident until no peer reads its shared
    // memory any more.
    int m0, mend, n0, bx0;
    place(first, m0, mend, n0, bx0);
    const int rpc = BM / p.ks, q = rpc / 4;  // rows, and groups of four, of this CTA
    const int ntok = min(p.bn, p.N - n0);
    const uint32_t red = smem_u32(smem);
    bool range_err = false;
    for (int i = threadIdx.x; i < q * ntok; i += THREADS) {
      const int t = i / q, rr = z * rpc + (i - t * q) * 4;
      const uint32_t off = red + (uint32_t)(t * BM + rr) * 4u;
      float4 a[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < p.ks) a[k] = ld_dsmem_f32x4(mapa_shared(off, (uint32_t)((z + k) & (p.ks - 1))));
      float f[4] = {a[0].x, a[0].y, a[0].z, a[0].w};
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (k < p.ks) {
          f[0] += a[k].x;
          f[1] += a[k].y;
          f[2] += a[k].z;
          f[3] += a[k].w;
        }
      const int tok = n0 + t, row = m0 + rr;
      uint16_t h[4], l[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kEpi != EPI_Y_ONLY) split_hl<kEpi>(f[j], h[j], l[j], range_err);
        if (row + j >= mend) continue;
        const int col = __ldg(p.cols + row + j);
        if ((unsigned)col >= (unsigned)p.m)
          latch_status(p.status, PIFA_ERR_DEVICE_INDEX);
        else
          p.Y[(int64_t)tok * p.ldy + col] = __float2bfloat16_rn(f[j]);
      }
      if (kEpi != EPI_Y_ONLY && row < p.ldyp) {  // rows beyond M hold zeros (padding columns)
        const int64_t o = (int64_t)tok * p.ldyp + row;
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(p.yp_hi) + o) =
            make_uint2((uint32_t)h[0] | (uint32_t)h[1] << 16, (uint32_t)h[2] | (uint32_t)h[3] << 16);
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(p.yp_lo) + o) =
            make_uint2((uint32_t)l[0] | (uint32_t)l[1] << 16, (uint32_t)l[2] | (uint32_t)l[3] << 16);
      }
    }
    if (range_err) latch_status(p.status, PIFA_ERR_RANGE);
    cluster_sync_all();
  }
}

using Kern = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const GemmArgs);

// How a GEMM is tiled: by pairs of CTAs (256 weight rows) or by one CTA (128), tokens per tile, and
// K-slices per tile (one-CTA tiles only: the CTAs of a cluster).
struct GemmShape {
  bool pair;
  int bn, ks;
};

Kern kernel_of(int epi, const GemmShape& sh) {
  static const Kern k[3][3] = {
      {pifa_umma_gemm<EPI_Y_ONLY, false, true>, pifa_umma_gemm<EPI_Y_ONLY, false, false>, pifa_umma_gemm<EPI_Y_ONLY, true, false>},
      {pifa_umma_gemm<EPI_SPLIT_BF16, false, true>, pifa_umma_gemm<EPI_SPLIT_BF16, false, false>,
       pifa_umma_gemm<EPI_SPLIT_BF16, true, false>},
      {pifa_umma_gemm<EPI_SPLIT_F16, false, true>, pifa_umma_gemm<EPI_SPLIT_F16, false, false>,
       pifa_umma_gemm<EPI_SPLIT_F16, true, false>}};
  return k[epi][sh.pair ? 0 : sh.ks > 1 ? 2 : 1];
}

// Tiles that run at once on the current device: pairs, single CTAs, clusters of 2 and of 4. A query that
// fails counts as one for this call and is made again by the next.
struct Slots {
  int pair, one, cl[2];
};
Slots tile_slots() {
  static std::mutex mu;
  static std::map<int, Slots> known;
  int dev = 0;
  bool ok = cudaGetDevice(&dev) == cudaSuccess;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = known.find(dev);
  if (ok && it != known.end()) return it->second;
  auto query = [&](const GemmShape& sh) {
    const Kern k = kernel_of(EPI_Y_ONLY, sh);
    cudaLaunchConfig_t cfg = {};
    const unsigned c = sh.pair ? 2u : (unsigned)sh.ks;
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = c;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n < 1) {
      n = 1;
      ok = false;
    }
    cudaGetLastError();  // a failed query leaves no sticky error behind
    return n;
  };
  const Slots s = {query({true, BNMAX, 1}), query({false, BNMAX, 1}), {query({false, BNMAX, 2}), query({false, BNMAX, 4})}};
  if (ok) known[dev] = s;
  return s;
}

// Bytes of one 64-column chunk of a tile in a CTA's ring, and chunks per stage: two where the ring
// holds at least six (a barrier hand-off per 128 columns instead of per 64 takes a fifth off the step
// of narrow tiles, but two stages in all would starve wide one-CTA ones).
uint32_t chunk_bytes(bool pair, int bn) { return A_BYTES + (uint32_t)(pair ? bn / 2 : bn) * BK * 2; }
int subs_for(bool pair, int bn) { return RING_BYTES / chunk_bytes(pair, bn) >= 6 ? 2 : 1; }

// The tiling of G groups of `rows` weight rows x T tokens that finishes first by the measured costs, in
// cycles: a chunk's (see the head of this file), an unhidden epilogue's 25 per token of a tile's width,
// a launch's 9600 (a pair's 10600), a cluster's 12500 and its exchange of partial tiles 20 per token. (An
// epilogue that hides only as far as the next tile's chunks last, and costs refitted to the 398 GEMMs named above,
// gained up to 15% on some drawn calls and lost up to 9% on others.)
GemmShape pick_shape(int64_t G, int64_t rows, int64_t T, int64_t kchunks) {
  const Slots slots = tile_slots();
  GemmShape best = {true, BNMAX, 1};
  double best_cost = -1.0;
  for (int form = 0; form < 4; ++form) {  // pairs, single CTAs, clusters of 2, of 4
    const bool pair = form == 0;
    const int ks = form < 2 ? 1 : form == 2 ? 2 : 4;
    if (ks > 1 && kchunks < 8 * ks) break;
    const int64_t mt = G * ((rows + (pair ? PM : BM) - 1) / (pair ? PM : BM));
    const int64_t at_once = form == 0 ? slots.pair : form == 1 ? slots.one : slots.cl[form - 2];
    for (int bn = T < BNMAX ? (int)(T + 31) / 32 * 32 : BNMAX; bn >= 32; bn -= 32) {
      const int64_t rounds = (mt * ((T + bn - 1) / bn) + at_once - 1) / at_once;
      const double step = pair ? 330.0 + 0.85 * bn : subs_for(false, bn) == 2 ? 410.0 + 0.3 * bn : 480.0 + 0.66 * bn;
      double cost = (double)rounds * (double)((kchunks + ks - 1) / ks) * step + 25.0 * bn;
      cost += ks > 1 ? (double)rounds * (12500.0 + 20.0 * bn) : pair ? 10600.0 : 9600.0;
      if (best_cost < 0.0 || cost < best_cost) {
        best_cost = cost;
        best = {pair, bn, ks};
      }
    }
  }
  return best;
}

int run_gemm(int epi, const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1, const GemmArgs& g,
             const GemmShape& sh, cudaStream_t stream) {
  const Kern kern = kernel_of(epi, sh);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e != cudaSuccess) return pifa_fail_cuda("cudaFuncSetAttribute(prefill gemm)", e);
  // programmatic dependent launch: each GEMM may start (weight tiles in flight) while the previous
  // kernel of the stream drains; its dependent loads follow griddepcontrol.wait
  cudaLaunchConfig_t cfg = {};
  const unsigned per = sh.pair ? 2u : (unsigned)sh.ks;  // CTAs per tile: a cluster
  const int at_once = sh.pair ? tile_slots().pair : sh.ks > 1 ? g.tiles : tile_slots().one;
  cfg.gridDim = dim3(per * (unsigned)(g.tiles < at_once ? g.tiles : at_once));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = per;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = pifa_launch_ex(&cfg, kern, a, b0, b1, g);
  if (e != cudaSuccess) return pifa_fail_cuda("prefill gemm launch", e);
  return PIFA_OK;
}

// Fills the tiling of an M x T GEMM (G groups of rows) into `g`.
int set_tiling(GemmArgs& g, int64_t G, int64_t M, int64_t T, const GemmShape& sh) {
  g.M = (int)M;
  g.N = (int)T;
  g.bn = sh.bn;
  g.ks = sh.ks;
  g.gsz = (int)(M / G);
  const int tm = sh.pair ? PM : BM;
  g.mtg = (g.gsz + tm - 1) / tm;
  g.mt = (int)G * g.mtg;
  g.nt = (int)((T + sh.bn - 1) / sh.bn);
  if ((int64_t)g.mt * g.nt * 4 >= ((int64_t)1 << 31))
    return pifa_fail(PIFA_ERR_UNSUPPORTED, "prefill: more than 2^30 tiles");
  g.tiles = g.mt * g.nt;
  g.subs = subs_for(sh.pair, sh.bn);
  g.ksteps = (g.kchunks + g.subs - 1) / g.subs;
  g.stage_bytes = (uint32_t)g.subs * chunk_bytes(sh.pair, sh.bn);
  g.stages = (int)(RING_BYTES / g.stage_bytes);
  if (g.stages > MAX_STAGES) g.stages = MAX_STAGES;
  // Walking token tiles first (when M > T) runs a weight-row block's tiles together, sharing its A
  // tile, with all of B (T x K) the round's other operand; walking row tiles first shares B tiles
  // with all of A (M x K): the round's working set is the smaller way round.
  g.tok_fast = M > T ? 1 : 0;
  return PIFA_OK;
}

inline int64_t pad8(int64_t v) { return (v + 7) / 8 * 8; }

}  // namespace

int64_t prefill_split_workspace_bytes(const PifaShape& s) {
  const int64_t one = ((s.T * pad8(s.groups * s.r) * 2 + 255) / 256) * 256;  // 2-byte T x pad8(G r)
  return 2 * one;  // hi and lo
}

int launch_prefill_split(const PifaShape& s, const PifaPointers& p, int* status, uint64_t timeout_ns,
                         cudaStream_t stream) {
  const bool f16 = s.c_dtype == PIFA_DTYPE_FP16;
  const int64_t G = s.groups;  // layers sharing X: GEMM 1 over their stacked pivot rows
  const int64_t ldyp = pad8(G * s.r);
  const int64_t one = ((s.T * ldyp * 2 + 255) / 256) * 256;
  void* hi = p.ws;
  void* lo = reinterpret_cast<uint8_t*>(p.ws) + one;

  CUtensorMap tWp, tX, tC, tHi, tLo;
  int st;
  GemmArgs g1 = {};
  g1.kchunks = (int)((s.n + BK - 1) / BK);
  g1.passes = 1;
  const GemmShape sh1 = pick_shape(1, G * s.r, s.T, g1.kchunks);
  const uint32_t box1 = (uint32_t)(sh1.pair ? sh1.bn / 2 : sh1.bn);
  if ((st = set_tiling(g1, 1, G * s.r, s.T, sh1)) != PIFA_OK) return st;
  if ((st = make_tmap_2d(&tWp, PIFA_DTYPE_BF16, p.Wp, G * s.r, s.n, s.ldwp, BK, BM)) != PIFA_OK) return st;
  if ((st = make_tmap_2d(&tX, PIFA_DTYPE_BF16, p.X, s.T, s.n, s.ldx, BK, box1)) != PIFA_OK) return st;
  g1.idesc = idesc_bf16_f32(sh1.pair ? PM : BM, (uint32_t)sh1.bn);
  g1.cols = p.piv;
  g1.m = (int)(G * s.m);
  g1.Y = reinterpret_cast<bf16*>(p.Y);
  g1.ldy = s.ldy;
  g1.yp_hi = hi;
  g1.yp_lo = lo;
  g1.ldyp = ldyp;
  g1.status = status;
  g1.timeout_ns = timeout_ns;
  if ((st = run_gemm(f16 ? EPI_SPLIT_F16 : EPI_SPLIT_BF16, tWp, tX, tX, g1, sh1, stream)) != PIFA_OK) return st;
  if (s.m == s.r) return PIFA_OK;

  GemmArgs g2 = g1;
  g2.kchunks = (int)((s.r + BK - 1) / BK);
  g2.passes = 2;
  const int64_t M2 = G * (s.m - s.r);
  const GemmShape sh2 = pick_shape(G, s.m - s.r, s.T, 2 * g2.kchunks);
  const uint32_t box2 = (uint32_t)(sh2.pair ? sh2.bn / 2 : sh2.bn), tm2 = sh2.pair ? PM : BM;
  // group g's non-pivot rows (no tile spans two groups) read the hi/lo columns [g r, (g + 1) r)
  if ((st = set_tiling(g2, G, M2, s.T, sh2)) != PIFA_OK) return st;
  g2.goff = G > 1 ? (int)s.r : 0;
  if ((st = make_tmap_2d(&tC, s.c_dtype, p.C, M2, s.r, s.ldc, BK, BM)) != PIFA_OK) return st;
  if ((st = make_tmap_2d(&tHi, s.c_dtype, hi, s.T, G * s.r, ldyp, BK, box2)) != PIFA_OK) return st;
  if ((st = make_tmap_2d(&tLo, s.c_dtype, lo, s.T, G * s.r, ldyp, BK, box2)) != PIFA_OK) return st;
  g2.idesc = f16 ? idesc_f16_f32(tm2, (uint32_t)sh2.bn) : idesc_bf16_f32(tm2, (uint32_t)sh2.bn);
  g2.cols = p.nonpiv;
  g2.yp_hi = nullptr;
  g2.yp_lo = nullptr;
  return run_gemm(EPI_Y_ONLY, tC, tHi, tLo, g2, sh2, stream);
}
