// a2 + a3 + a4 in one launch: importance scores (Eq. 4), exact selection of the entries to evict
// (Alg. 1, Evict) and hole-fill compaction back to the budget M (the last step of Alg. 1's loop body).
//
// One thread-block cluster of Cn CTAs per (kv-head, layer).
//   phase 1 (MODE = kScoreAttention, bf16)  the 128-key tiles of the candidates are dealt round-robin to the CTAs
//            of the cluster.  Per tile: K tile by TMA, S^T = K_tile Q_obs^T on the tensor cores (keys on
//            the TMEM lanes, observer rows on the columns), each thread sums 2^(s*scale - lse2) over
//            the observer columns of its key and writes the score.  Two tiles are in flight per CTA
//            (two K buffers, two TMEM accumulators, two epilogue warp groups).
//            MODE = kScoresGiven: the scores are already in the workspace (score kernel of its own).
//            MODE = kScoreKeyDiff: query-agnostic score 1 - cos(k_j, mean key) (Sec. 3.2), any dtype.
//   phase 2  cluster barrier; then EVERY CTA reads all scores of its kv-head (L2-resident), builds the
//            64-bit keys in shared memory and runs the same exact selection redundantly -- cheaper than
//            a distributed histogram, since the SM-to-SM path is narrow and the other SMs would idle.
//   phase 3  every CTA derives the same ordered hole / survivor lists and executes every Cn-th move.
// Entry j gets the key (score bits << 32) | ~pos: a larger key means a higher score and, at equal
// score, an older entry; keys are unique where positions are.  Scores are sums of probabilities,
// hence >= 0, so their IEEE bit patterns order like integers.  The n_keep-th largest key (the cut-off)
// is found exactly by an MSB-first radix descent with 11-bit digits that starts below the bits all
// keys share and stops as soon as the bin that holds the cut-off survives as a whole.  Where a caller repeats positions
// and equal keys lie across the cut-off, the first of them in row order stay.
#pragma once
#include <cuda.h>
#include <type_traits>
#include "geom.cuh"
#include "ptx.cuh"

namespace kvc {

// 512 threads and, with up to 128 observer rows, at most 97 KB of shared memory per CTA: two CTAs share an SM, so that one
// scores (TMA / tensor-core bound) while the other selects (barrier bound) when many kv-heads are in flight.  With more
// rows a CTA asks for up to 129 KB and is alone on its SM.
static constexpr int kCompressThreads = 512;
static constexpr int kDigitBits = 11;
static constexpr int kSelBins = 1 << kDigitBits;
static constexpr int kRankMax = 256;          // keys of the cut-off bin that are ranked directly instead of by further rounds
// Candidates up to which all are ranked directly: 48 candidates 6.1 -> 5.2 us, 96 4.3 -> 3.6; 160 4.3 -> 4.5, hence the line.
static constexpr int kDirectMax = 128;
static constexpr int kMaxKeysSmem = 6144;     // candidates whose keys fit the shared-memory table (48 KB)
static constexpr int kMaxMovesSmem = 2048;    // moves whose (src, dst) fit the shared-memory tables (16 KB)
// observer rows (w * G) the fused scoring phase takes: up to 128, or up to 256 with a CTA alone on its SM
static constexpr int kMaxObsRowsFused = 128, kMaxObsRowsWide = 256;
static constexpr int kMaxClusterWide = 16;   // largest cluster the host asks for (non-portable size: more than 8 CTAs)
static constexpr int kScoresGiven = 0, kScoreAttention = 1, kScoreKeyDiff = 2;   // what phase 1 of compress_kernel does
static constexpr int kSubTileBytesC = 128 * 128;

__device__ __forceinline__ unsigned long long select_key(float score, int pos) {
  return (static_cast<unsigned long long>(__float_as_uint(score)) << 32) |
         static_cast<unsigned long long>(0xFFFFFFFFu - static_cast<uint32_t>(pos));
}

// The selection and the listing run on the whole block (measured: a quarter of it pays less per barrier but more
// per key, and loses).
static constexpr int kTeam = kCompressThreads;

struct CompressSmem {
  uint64_t q_full, k_full[2], s_full[2], t_free[2];
  uint32_t tmem_base;
  int wait_ctl[2];           // [0] abort flag, [1] wait limit in units of 1024 cycles (see mbar_wait)
  alignas(16) float lse2[256];
  unsigned long long list[2 * (kTeam / 32) + 2];
  int scan_scratch[kTeam / 32 + 1];
  unsigned long long s_prefix, cutoff, tie_key;
  int s_remaining, s_bin_count, s_count, row_cut;
};

// grid (Cn, Hkv, nl), cluster (Cn,1,1), block 512.
// dynamic smem: the larger of the scoring buffers (two K tiles + OBS observer rows) and of the key
// and move tables with the two histograms (80 KB), + 1 KB.
// What bounds it: latency -- a chain of block barriers and L2 round trips -- and, since most of its code runs once per
// launch, instruction fetch: block-wide sums by one redux per warp instead of unrolled loops over the warps' totals and
// six loads per step instead of twelve take the kernel from 7.4 to 6.8 us (32 kv-heads x 288 candidates), 5.2 to 4.4
// (1 x 160) and 10.8 to 10.2 (8 x 2212).
template <int D, int MODE, int OBS>
__global__ void __launch_bounds__(kCompressThreads, 2) compress_kernel(const __grid_constant__ CUtensorMap tm_k,
                                                                       const __grid_constant__ CUtensorMap tm_qobs,
                                                                       const __grid_constant__ CUtensorMap tm_kin,
                                                                       const char* __restrict__ kin, char* __restrict__ cache, char* __restrict__ ws,
                                                                       Geom p, int Cn, int elem_bytes) {
  constexpr int NSUB = D / 64;
  constexpr int K_TILE_BYTES = NSUB * kSubTileBytesC;
  constexpr int kQSubBytes = OBS * 128;                // OBS observer rows x 128 B
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ CompressSmem sh;

  const int layer = blockIdx.z, g = blockIdx.y;
  const int rank = Cn > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  char* blob = cache + layer * p.cache_ls;
  int* pos = reinterpret_cast<int*>(blob + p.pos_off) + static_cast<long long>(g) * p.cap;
  char* slot = ws_slot(ws, p, layer);
  float* score = reinterpret_cast<float*>(slot + p.score_off) + static_cast<long long>(g) * p.cap;
  int* msrc_g = reinterpret_cast<int*>(slot + p.msrc_off) + static_cast<long long>(g) * p.max_chunk;
  int* mdst_g = reinterpret_cast<int*>(slot + p.mdst_off) + static_cast<long long>(g) * p.max_chunk;
  int* mcount = reinterpret_cast<int*>(slot + p.mcount_off);
  volatile int* abort_flag = sh.wait_ctl;
  if (tid == 0) { sh.wait_ctl[0] = 0; sh.wait_ctl[1] = p.wait_limit_k; }
  // The next kernel of the stream may set itself up meanwhile -- once this one has its tensor memory: a dependent that
  // allocates some in front of its own dependency wait could otherwise take what this CTA still needs, and both would wait.
  // (Allocating first, in this warp alone, keeps the trigger early: image request 2736 -> 2755 us, behind the block's first
  // barrier 2759.)
  if constexpr (MODE == kScoreAttention) {
    if (warp == 8) {
      tmem_alloc(&sh.tmem_base, 2 * OBS);
      tmem_relinquish();
      pdl_launch_dependents();
    }
  } else {
    pdl_launch_dependents();
  }
  // Before the dependency wait this kernel may read what was complete before the attention kernel of the same call began
  // its work: the call's inputs and the cache rows below n_c = n_sc (on a side stream, where the caller may reuse k by now,
  // n_sc covers all rows and there is nothing to wait for).  The attention kernel allows this launch only after its own
  // wait, so everything that precedes it in the stream has finished and is in L2; these reads go there (TMA, ld.global.cg)
  // and never through L1, which is only known to be current behind this kernel's own wait.  What it writes before the wait
  // are the scores, move lists and counts of its workspace slot: the attention touches none of them, and the kernels that
  // used the slot before had finished when the attention was past its own wait.  Cache rows are written behind the wait only.
  // (Loads and products then overlap the attention's end: 32 kv-heads x 288 candidates 7.0 -> 6.4 us behind the wait,
  // 4 x 2300 x 224 observer rows 11.6 -> 10.6.  The query-agnostic policy has all but the moves there, see below.)

  // ------------------------------------------------------------------------------------ phase 1: scores
  if constexpr (MODE == kScoreAttention) {
    uint8_t* sK = smem;                              // two K tiles
    uint8_t* sQ = smem + 2 * K_TILE_BYTES;           // observer rows
    // Key tiles: the cache rows [0, n_sc), then the block's own tokens read from the k input, as in the attention kernel.
    // Neither depends on the attention kernel, and both are complete when this kernel starts (see below): K, Q and the
    // products come before the dependency wait, only the exponentials need the log-sum-exp behind it.
    const int cache_tiles = (p.n_sc + 127) / 128, n_tiles = cache_tiles + (p.n_cand - p.n_sc + 127) / 128;
    const int my_tiles = rank < n_tiles ? (n_tiles - rank + Cn - 1) / Cn : 0;
    const int cols = p.w * p.G;                      // observer columns (<= OBS: one MMA, two accumulators of OBS columns)
    const int n_mma = (cols + 15) & ~15;
    if (tid == 0) {
      mbar_init(&sh.q_full, 1);
      for (int i = 0; i < 2; ++i) { mbar_init(&sh.k_full[i], 1); mbar_init(&sh.s_full[i], 1); mbar_init(&sh.t_free[i], 4); }
      mbar_fence_init();
    }
    // observer rows beyond the real ones are padding: keep them finite
    for (int i = tid; i < NSUB * kQSubBytes / 16; i += kCompressThreads) reinterpret_cast<uint4*>(sQ)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sh.tmem_base;
    if (warp == 8) {
      if (lane == 0) {
        tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_qobs); tma_prefetch_desc(&tm_kin);
        if (p.stamp_early) stamp_begin(p);
        bool ok = true;
        auto load_tile = [&](int i) {                  // tile i of this CTA into K buffer i & 1
          const int b = i & 1, kt = rank + i * Cn;
          mbar_expect_tx(&sh.k_full[b], K_TILE_BYTES);
          for (int sub = 0; sub < NSUB; ++sub) {
            void* dst = sK + b * K_TILE_BYTES + sub * kSubTileBytesC;
            if (kt < cache_tiles) tma_load_4d(dst, &tm_k, &sh.k_full[b], sub * 64, kt * 128, g, layer);
            else tma_load_4d(dst, &tm_kin, &sh.k_full[b], sub * 64, g, (kt - cache_tiles) * 128, layer);
          }
        };
        if (my_tiles > 0) {
          mbar_expect_tx(&sh.q_full, NSUB * p.w * p.G * 128);
          for (int sub = 0; sub < NSUB; ++sub)
            tma_load_4d(sQ + sub * kQSubBytes, &tm_qobs, &sh.q_full, sub * 64, g * p.G, p.n - p.w, layer);
          for (int i = 0; i < my_tiles && i < 2; ++i) load_tile(i);
          ok = mbar_wait(&sh.q_full, 0, abort_flag);
        }
        const uint32_t idesc = idesc_bf16_f32(128, n_mma, 0, 0);
        constexpr uint32_t hi = smem_desc_hi_sw128(1024);
        const uint32_t k_lo0 = smem_desc_lo(smem_u32(sK), 16), q_lo = smem_desc_lo(smem_u32(sQ), 16);
        int i = 0;
        for (; i < my_tiles && ok; ++i) {
          const int b = i & 1;
          ok = mbar_wait(&sh.k_full[b], (i >> 1) & 1, abort_flag);
          if (ok && i >= 2) ok = mbar_wait(&sh.t_free[b], ((i - 2) >> 1) & 1, abort_flag);   // accumulator b read out
          if (!ok) break;
          tc_fence_after_sync();
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            mma_ss_lh(tmem + b * OBS, k_lo0 + ((b * K_TILE_BYTES + (kk / 4) * kSubTileBytesC + (kk % 4) * 32) >> 4), hi,
                      q_lo + (((kk / 4) * kQSubBytes + (kk % 4) * 32) >> 4), hi, idesc, kk > 0);
          mma_commit(&sh.s_full[b]);
          if (i + 2 < my_tiles) {                    // refill K buffer b once the MMAs that read it are done
            ok = mbar_wait(&sh.s_full[b], (i >> 1) & 1, abort_flag);
            if (!ok) break;
            load_tile(i + 2);
          }
        }
        // What follows the block's barrier lays the selection's tables over the tiles: not before the loads that nobody has waited
        // for are complete, those of the observer rows and of tiles i and i + 1.  (This and the wait in front of the release of TMEM:
        // image 2643 -> 2648 us, image from a graph 1475 -> 1481, video 7838 -> 7850.)
        if (__builtin_expect(!ok, 0)) {
          mbar_drain(&sh.q_full, 0);
#pragma unroll 1
          for (int j = i; j < min(i + 2, my_tiles); ++j) mbar_drain(&sh.k_full[j & 1], (j >> 1) & 1);
        }
      }
      __syncwarp();
    } else if (warp < 8) {
      const int b = warp >> 2;
      const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
      pdl_wait();
      if (tid == 0) stamp_begin(p);
      const float* lse = reinterpret_cast<const float*>(slot + p.lse_off);
      // log-sum-exp of the observer rows in log2 units; padding columns get +inf (2^-inf = 0).
      // Each epilogue group fills the whole table (same values), so no cross-group barrier is needed.
      for (int c = (warp & 3) * 32 + lane; c < 256; c += 128) {
        float lv = INFINITY;
        if (c < cols) lv = lse[static_cast<long long>(p.n - p.w + c / p.G) * p.Hq + g * p.G + c % p.G] * 1.4426950408889634f;
        sh.lse2[c] = lv;
      }
      named_barrier(1 + b, 128);
      bool ok = true;
      for (int i = b; i < my_tiles; i += 2) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.s_full[b], (i >> 1) & 1, abort_flag));
        if (!ok) break;
        tc_fence_after_sync();
        float acc = 0.f;
        float acc2 = 0.f;
        for (int c0 = 0; c0 < n_mma; c0 += 32) {       // n_mma is a multiple of 16: the second half may be absent
          uint32_t sr[32];
          const bool two = c0 + 16 < n_mma;
          tmem_ld16(tmem + b * OBS + lane_addr + c0, sr);
          if (two) tmem_ld16(tmem + b * OBS + lane_addr + c0 + 16, sr + 16);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 16; ++k) acc += fast_exp2(fmaf(__uint_as_float(sr[k]), p.scale_log2, -sh.lse2[c0 + k]));
          if (two) {
#pragma unroll
            for (int k = 16; k < 32; ++k) acc2 += fast_exp2(fmaf(__uint_as_float(sr[k]), p.scale_log2, -sh.lse2[c0 + k]));
          }
        }
        acc += acc2;
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.t_free[b]);              // one arrival per warp of the epilogue group
        const int kt = rank + i * Cn, row = (warp & 3) * 32 + lane;
        const int key = kt < cache_tiles ? kt * 128 + row : p.n_sc + (kt - cache_tiles) * 128 + row;
        if (key < (kt < cache_tiles ? p.n_sc : p.n_cand)) score[key] = acc;
      }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 8) {
      // The warps that read TMEM may have given up waiting for MMAs under way.  (One more phase of q_full, which is done with.)
      if (__builtin_expect(abort_flag[0] != 0, 0) && lane == 0) {
        mma_commit(&sh.q_full);
        mbar_drain(&sh.q_full, 1);
      }
      __syncwarp();
      tc_fence_after_sync();
      tmem_dealloc(tmem, 2 * OBS);
    }
  } else if constexpr (MODE == kScoreKeyDiff) {
    // Query-agnostic score (Sec. 3.2): anchor mu = mean of the tot keys the cache holds after the append,
    // score_j = max(0, 1 - cos(k_j, mu)) for the candidates (>= 0, so its bit pattern orders like an integer; a
    // zero key or anchor has cosine 0).  A row is read by lpr lanes of 16 bytes; the CTAs of the cluster take the 128-row
    // tiles round-robin, add their partial sums through distributed shared memory, and every CTA scores its own tiles
    // (second read of K: L2).  The order of every sum is fixed by the cluster size alone.
    // Bound: latency and instruction fetch.  4 kv-heads x 1833 keys, d = 64: the kernel 13.6 -> 9.8 us (8 x 5120, d = 128
    // 23.9 -> 19.2) with loads in flight across tiles, the remote sums fetched together
    // (one at a time each costs a round trip), no array in local memory, one lane per row finishing its score, and the
    // shorter selection.  (Fetching the share into shared memory with bulk copies, or keeping it in registers: no faster.)
    float* s_part = reinterpret_cast<float*>(smem);                 // [16 warps][d] partial sums
    float* s_sum = s_part + (kCompressThreads / 32) * 128;         // [d] this CTA's sum (read by the cluster)
    float* s_mu = s_sum + 128;                                      // [d] the anchor
    if (tid == 0 && p.stamp_early) stamp_begin(p);
    const int d = p.d, epl = 16 / elem_bytes;                       // elements per 16-byte piece: 8 (bf16) or 4 (fp32)
    const int lpr = d / epl, rpw = 32 / lpr;                        // lanes per row, rows per warp and step
    const int sub = lane / lpr, piece = lane % lpr;
    const long long row_bytes = static_cast<long long>(d) * elem_bytes;
    const char* Kg = blob + static_cast<long long>(g) * p.cap * row_bytes + piece * 16;
    const char* Kn = kin + (layer * p.kv_ls + static_cast<long long>(g) * d) * elem_bytes + piece * 16;
    auto fetch = [&](int row) {                                     // (the block's rows from the input, as above; through L2)
      return __ldcg(reinterpret_cast<const uint4*>(row < p.n_sc ? Kg + row * row_bytes : Kn + (row - p.n_sc) * p.Hkv * row_bytes));
    };
    auto widen = [&](const uint4 raw, float* f) {
      if (elem_bytes == 2) {
        const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w4[i] << 16); f[2 * i + 1] = __uint_as_float(w4[i] & 0xffff0000u); }
      } else {
        f[0] = __uint_as_float(raw.x); f[1] = __uint_as_float(raw.y); f[2] = __uint_as_float(raw.z); f[3] = __uint_as_float(raw.w);
#pragma unroll
        for (int i = 4; i < 8; ++i) f[i] = 0.f;
      }
    };
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    constexpr int kRowsInFlight = 4;                               // independent loads per lane
    const int rstep = (kCompressThreads / 32) * rpw;               // rows the CTA covers per step
    const int tiles_all = (p.tot + 127) / 128, my_tiles = rank < tiles_all ? (tiles_all - rank + Cn - 1) / Cn : 0;
    const int log_steps = __ffs(128 / rstep) - 1, n_steps = my_tiles << log_steps;   // steps per tile: 2, 4 or 8
    auto row_of = [&](int i) { return (rank + (i >> log_steps) * Cn) * 128 + warp * rpw + sub + (i & ((1 << log_steps) - 1)) * rstep; };
    uint4 raw[kRowsInFlight];
    auto load = [&](int i0) {
#pragma unroll
      for (int u = 0; u < kRowsInFlight; ++u) {
        const int row = row_of(i0 + u);
        raw[u] = i0 + u < n_steps && row < p.tot ? fetch(row) : make_uint4(0u, 0u, 0u, 0u);
      }
    };
#pragma unroll 1
    for (int i0 = 0; i0 < n_steps; i0 += kRowsInFlight) {
      load(i0);
#pragma unroll
      for (int u = 0; u < kRowsInFlight; ++u) {
        float f[8];
        widen(raw[u], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += f[e];
      }
    }
    for (int o = lpr; o < 32; o <<= 1) {
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    }
    if (sub == 0)
#pragma unroll
      for (int e = 0; e < 8; ++e)                                   // (a run-time bound would put acc in local memory)
        if (e < epl) s_part[warp * 128 + piece * epl + e] = acc[e];
    __syncthreads();
    if (tid < d) {
      float t = 0.f;
      for (int w2 = 0; w2 < kCompressThreads / 32; ++w2) t += s_part[w2 * 128 + tid];
      s_sum[tid] = t;
    }
    __syncthreads();
    if (Cn > 1) { cluster_arrive(); cluster_wait(); }
    if (tid < d) {
      float t = 0.f;
      if (Cn > 1) {
        const uint32_t a = smem_u32(&s_sum[tid]);
        float part[kMaxClusterWide];
#pragma unroll
        for (int rk = 0; rk < kMaxClusterWide; ++rk) part[rk] = rk < Cn ? dsmem_ld_f32(dsmem_addr(a, rk)) : 0.f;
#pragma unroll
        for (int rk = 0; rk < kMaxClusterWide; ++rk) t += part[rk];
      } else {
        t = s_sum[tid];
      }
      s_mu[tid] = t / static_cast<float>(p.tot);
    }
    __syncthreads();
    float mu[8], mu_norm = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) mu[e] = e < epl ? s_mu[piece * epl + e] : 0.f;
    for (int i = lane; i < d; i += 32) mu_norm += s_mu[i] * s_mu[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mu_norm += __shfl_xor_sync(0xffffffffu, mu_norm, o);
    mu_norm = sqrtf(mu_norm);
#pragma unroll 1
    for (int i0 = 0; i0 < n_steps; i0 += kRowsInFlight) {
      load(i0);
      float dot[kRowsInFlight], nrm[kRowsInFlight];
#pragma unroll
      for (int u = 0; u < kRowsInFlight; ++u) {
        float f[8];
        widen(raw[u], f);
        dot[u] = nrm[u] = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) { dot[u] = fmaf(f[e], mu[e], dot[u]); nrm[u] = fmaf(f[e], f[e], nrm[u]); }
      }
      for (int o = 1; o < lpr; o <<= 1) {
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) {
          dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
          nrm[u] += __shfl_xor_sync(0xffffffffu, nrm[u], o);
        }
      }
      // lane `piece` of a row group finishes row `piece` of the batch (every lane holds all sums)
      float dt = dot[0], nm = nrm[0];
#pragma unroll
      for (int u = 1; u < kRowsInFlight; ++u)
        if (piece == u) { dt = dot[u]; nm = nrm[u]; }
      const int r = row_of(i0 + piece);
      // fp32 rounding can put the cosine of a key (nearly) parallel to the anchor a little above 1: clamp, so
      // that the score stays >= 0 and select_key's ordering by bit pattern holds
      const float den = sqrtf(nm) * mu_norm;
      if (piece < kRowsInFlight && i0 + piece < n_steps && r < p.n_cand) score[r] = den > 0.f ? fmaxf(0.f, 1.f - dt / den) : 1.f;
    }
  } else {
    if (tid == 0) { pdl_wait(); stamp_begin(p); }
    __syncthreads();
  }
  if (Cn > 1) {                                       // every score of this kv-head is in the workspace
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }

  // ------------------------------------------------------------------------------------ phase 2: selection
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem);           // 48 KB
  int* tab_src = reinterpret_cast<int*>(smem + kMaxKeysSmem * 8);                    // 8 KB
  int* tab_dst = tab_src + kMaxMovesSmem;                                            // 8 KB
  // histograms of two consecutive rounds (the second doubles as the list of the last bin's keys): 2 x 8 KB
  int (*hists)[kSelBins] = reinterpret_cast<int (*)[kSelBins]>(smem + kMaxKeysSmem * 8 + 2 * kMaxMovesSmem * 4);
  const bool keys_in_smem = p.n_cand <= kMaxKeysSmem;
  // Position of candidate j.  The query-agnostic policy is still in front of the dependency wait here: the positions of the
  // cached entries come through L2, the attention kernel has yet to write those of the block's.
  auto pos_of = [&](int j) -> int {
    if constexpr (MODE == kScoreKeyDiff) return j < p.n_sc ? __ldcg(pos + j) : static_cast<int>(p.pos0 + (j - p.n_sc));
    else return pos[j];
  };
  // One pass builds the keys (six independent loads in flight per thread: the scores come from L2), folds the
  // AND and the OR of all keys -- the bits above the highest bit in which any two keys differ are common to all of
  // them (scores of similar magnitude share their exponent bits), and the descent starts below them, so that the
  // first digit already spreads the keys over many bins -- and clears the first histogram.
  unsigned long long k_and = ~0ull, k_or = 0ull;
  constexpr int kKeyLoads = 6;                                   // independent (score, position) loads in flight per thread
  for (int j0 = tid; j0 < p.n_cand; j0 += kKeyLoads * kCompressThreads) {
    float sc[kKeyLoads];
    int ps[kKeyLoads];
#pragma unroll
    for (int u = 0; u < kKeyLoads; ++u) {
      const int j = j0 + u * kCompressThreads;
      if (j < p.n_cand) { sc[u] = __ldcg(score + j); ps[u] = pos_of(j); }
    }
#pragma unroll
    for (int u = 0; u < kKeyLoads; ++u) {
      const int j = j0 + u * kCompressThreads;
      if (j < p.n_cand) {
        const unsigned long long k = select_key(sc[u], ps[u]);
        if (keys_in_smem) keys[j] = k;
        k_and &= k; k_or |= k;
      }
    }
  }
  {
    const unsigned a_lo = __reduce_and_sync(0xffffffffu, static_cast<unsigned>(k_and)), a_hi = __reduce_and_sync(0xffffffffu, static_cast<unsigned>(k_and >> 32));
    const unsigned o_lo = __reduce_or_sync(0xffffffffu, static_cast<unsigned>(k_or)), o_hi = __reduce_or_sync(0xffffffffu, static_cast<unsigned>(k_or >> 32));
    if (lane == 0) { sh.list[warp] = (static_cast<unsigned long long>(a_hi) << 32) | a_lo; sh.list[kTeam / 32 + warp] = (static_cast<unsigned long long>(o_hi) << 32) | o_lo; }
  }
  for (int i = tid; i < kSelBins; i += kTeam) hists[0][i] = 0;
  if (tid == 0) { sh.cutoff = ~0ull; sh.tie_key = 0ull; }
  __syncthreads();
  // Selection and listing exist twice, for keys in shared memory and for keys re-read from the workspace: with the
  // choice made per access the compiler issues the global loads of the second form in both cases.
  const int n_lo = min(p.B, p.tot);
  const int max_moves = min(p.n, p.tot - p.B);                   // at most this many entries sit at or above row B
  const bool tabs_in_smem = max_moves <= kMaxMovesSmem;
  int* msrc = tabs_in_smem ? tab_src : msrc_g;                   // with global tables every CTA writes all entries
  int* mdst = tabs_in_smem ? tab_dst : mdst_g;                   // itself (same values) and reads only its own writes
  auto select_and_list = [&](auto in_smem) {
  constexpr bool kInSmem = decltype(in_smem)::value;
  auto key_of = [&](int j) -> unsigned long long {
    if constexpr (kInSmem) return keys[j];
    else return select_key(__ldcg(score + j), pos_of(j));
  };
  unsigned long long thr = ~0ull;                                // n_keep == 0: nothing among the candidates survives
  int surplus = 0, row_cut = p.n_cand;                           // of the keys equal to thr, the last `surplus` rows do not survive
  // `ge` keys are at least as large as a thread's own, `rank` of them survive: the cut-off is the key with as many.  Nobody has
  // it if equal keys lie across the cut-off; then it is the largest key with more.
  // (Requests cost up to 0.5 % for it: image 2731 -> 2741 us, proxies 1790 -> 1798, the others within their noise.  Counting
  // survivors against holes in the listing instead: 0.5 - 2.7 %, a matter of code size.)
  auto cut_at = [&](unsigned long long my, int ge, int rank) {
    if (ge == rank) sh.cutoff = my;
    __syncthreads();
    thr = sh.cutoff;
    if (thr == ~0ull) {
      if (ge > rank) atomicMax(&sh.tie_key, my);
      __syncthreads();
      thr = sh.tie_key;
      if (my == thr) sh.s_count = ge - rank;
      __syncthreads();
      surplus = sh.s_count;
    }
  };
  if (kInSmem && p.n_keep > 0 && p.n_cand <= kDirectMax) {
    // few candidates: rank all of them (the bits they share, a histogram round and the list would cost more)
    unsigned long long my = 0ull;
    int ge = 0;
    if (tid < p.n_cand) {
      my = keys[tid];
      int i = 0;
#pragma unroll 4
      for (; i + 1 < p.n_cand; i += 2) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(keys + i);
        ge += (x.x >= my) + (x.y >= my);
      }
      if (i < p.n_cand) ge += keys[i] >= my;
    }
    cut_at(my, ge, p.n_keep);
  } else if (p.n_keep > 0) {
    {                                                            // (every thread: the same values)
      static_assert(kTeam == 512, "sixteen ANDs and sixteen ORs, one per lane");
      const unsigned long long x = sh.list[lane];
      const unsigned lo = static_cast<unsigned>(x), hi = static_cast<unsigned>(x >> 32);
      const bool ors = lane >= 16;
      k_and = (static_cast<unsigned long long>(__reduce_and_sync(0xffffffffu, ors ? ~0u : hi)) << 32) | __reduce_and_sync(0xffffffffu, ors ? ~0u : lo);
      k_or = (static_cast<unsigned long long>(__reduce_or_sync(0xffffffffu, ors ? hi : 0u)) << 32) | __reduce_or_sync(0xffffffffu, ors ? lo : 0u);
    }
    const unsigned long long differ = k_and ^ k_or;             // != 0: at least two distinct keys (n_cand > n_keep >= 1)
    const int top = 63 - __clzll(static_cast<long long>(differ));
    int shift = top >= kDigitBits - 1 ? top - (kDigitBits - 1) : 0, bits = top - shift + 1;
    // state of the descent, the same in every thread: the bits decided so far and the rank (1-based, from the top) of
    // the cut-off among the keys that share them
    unsigned long long prefix = top == 63 ? 0ull : (k_or >> (top + 1)) << (top + 1);
    int remaining = p.n_keep, hb = 0;
    while (true) {
      int* hist = hists[hb];
      const int hi = shift + bits;           // bits [hi, 64) are already decided
      for (int j = tid; j < p.n_cand; j += kTeam) {
        const unsigned long long key = key_of(j);
        if (hi >= 64 || (key >> hi) == (prefix >> hi)) atomicAdd(&hist[(key >> shift) & ((1u << bits) - 1)], 1);
      }
      for (int i = tid; i < kSelBins; i += kTeam) hists[hb ^ 1][i] = 0;   // for the next round
      __syncthreads();
      // descending scan: thread t owns the BPT bins from kSelBins - 1 - BPT*t downwards; scan inside the warp by
      // shuffles, across the warps by reading the totals of the warps before (one barrier)
      constexpr int BPT = kSelBins / kTeam;
      const int b0 = kSelBins - 1 - BPT * tid;
      int mine = 0;
#pragma unroll
      for (int i = 0; i < BPT; ++i) mine += hist[b0 - i];
      int incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) sh.scan_scratch[warp] = incl;
      __syncthreads();
      incl += __reduce_add_sync(0xffffffffu, lane < warp ? sh.scan_scratch[lane] : 0);
      int excl = incl - mine;
      if (excl < remaining && remaining <= incl) {               // the cut-off lies in one of my bins
        int b = b0, h = hist[b0];
        while (excl + h < remaining) { excl += h; --b; h = hist[b]; }
        sh.s_prefix = prefix | (static_cast<unsigned long long>(b) << shift);
        sh.s_remaining = remaining - excl;                       // rank inside the chosen bin, 1-based
        sh.s_bin_count = h;
        sh.s_count = 0;
      }
      __syncthreads();
      prefix = sh.s_prefix; remaining = sh.s_remaining;
      const int h = sh.s_bin_count;
      // Done when every bit is decided, or when the whole bin survives (its rank equals its size): then
      // the prefix with zeros below it separates the retained keys from the others.
      if (shift == 0 || remaining == h) { thr = prefix; surplus = h - remaining; break; }
      if (h <= kRankMax) {
        // few keys left in the cut-off bin: list them and rank them directly instead of descending further
        unsigned long long* lst = reinterpret_cast<unsigned long long*>(hists[hb ^ 1]);
        for (int j = tid; j < p.n_cand; j += kTeam) {
          const unsigned long long key = key_of(j);
          if ((key >> shift) == (prefix >> shift)) lst[atomicAdd(&sh.s_count, 1)] = key;
        }
        __syncthreads();
        unsigned long long my = 0ull;
        int ge = 0;
        if (tid < h) {
          my = lst[tid];
          for (int i = 0; i < h; ++i) ge += lst[i] >= my;
        }
        cut_at(my, ge, remaining);
        break;
      }
      bits = shift >= kDigitBits ? kDigitBits : shift;
      shift -= bits;
      hb ^= 1;
    }
  }
  if (surplus > 0) {                                             // rare: one warp looks for the rows, the last ones first
    if (warp == 0) {
      int left = surplus, first = p.n_cand;
      for (int j0 = p.n_cand - 1; left > 0 && j0 >= 0; j0 -= 32) {
        const int j = j0 - lane;
        const unsigned eq = __ballot_sync(0xffffffffu, j >= 0 && key_of(max(j, 0)) == thr);
        if ((eq >> lane & 1) && __popc(eq & ((1u << lane) - 1)) < left) {
          if constexpr (kInSmem) keys[j] = 0ull;                 // below every other key
          else first = j;
        }
        left -= __popc(eq);
      }
      if constexpr (!kInSmem) {
        first = __reduce_min_sync(0xffffffffu, first);
        if (lane == 0) sh.row_cut = first;
      }
    }
    __syncthreads();
    if constexpr (!kInSmem) row_cut = sh.row_cut;
  }

  // ------------------------------------------------------------------------------------ phase 3: compaction
  // holes: evicted entries in rows [0, B); survivors: retained entries in rows [B, tot), both in ascending
  // row order.  Entry j is retained iff it is protected (j >= n_cand) or its key >= thr.
  {
    // Every thread owns a run of consecutive rows: it counts its holes (rows below B) and survivors (rows from B
    // on), one scan over the block (shuffles inside the warps, one barrier across them) turns the counts into
    // offsets, and a second walk over the same rows writes the row indices, in ascending order.
    const int rpt = (p.tot + kTeam - 1) / kTeam;                 // rows per thread
    const int r0 = min(tid * rpt, p.tot), r1 = min(r0 + rpt, p.tot);
    auto retained = [&](int j) {
      if constexpr (kInSmem) return j >= p.n_cand || key_of(j) >= thr;
      if (j >= p.n_cand) return true;
      const unsigned long long key = key_of(j);
      return key > thr || (key == thr && j < row_cut);
    };
    unsigned long long mine = 0;                                  // holes in the low word, survivors in the high word
    for (int j = r0; j < r1; ++j) {
      const bool keep = retained(j);
      if (j < n_lo) mine += keep ? 0ull : 1ull;
      else mine += keep ? (1ull << 32) : 0ull;
    }
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sh.list[warp] = incl;
    __syncthreads();
    const unsigned long long tw = lane < kTeam / 32 ? sh.list[lane] : 0ull, prev = lane < warp ? tw : 0ull, own = incl - mine;
    int off_h = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(prev)) + static_cast<unsigned>(own));
    int off_s = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(prev >> 32)) + static_cast<unsigned>(own >> 32));
    const int total_holes = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(tw)));
    for (int j = r0; j < r1; ++j) {
      const bool keep = retained(j);
      if (j < n_lo) { if (!keep) mdst[off_h++] = j; }
      else if (keep) msrc[off_s++] = j;
    }
    if (tid == 0) sh.s_remaining = total_holes;                  // == number of survivors: the cache returns to B
  }
  };
  if (keys_in_smem) select_and_list(std::true_type{}); else select_and_list(std::false_type{});
  __syncthreads();
  const int total_holes = sh.s_remaining;
  if (rank == 0 && tid == 0) mcount[g] = total_holes;
  // The query-agnostic score, selection and listing need nothing of the attention kernel and are done in front of the wait;
  // the moves write rows that it reads.  (Behind the wait, mean of the 72 evicting calls of a request with up to 4 kv-heads x
  // 1801 candidates, d = 64: 6.4 us with the score alone in front of it, 1.6 with all three; the request 1577 -> 1278 us.)
  if constexpr (MODE == kScoreKeyDiff) {
    pdl_wait();
    if (tid == 0) stamp_begin(p);
  }
  if (Cn > 1) {                                                  // the moves overwrite positions (and rows) that the
    cluster_arrive_relaxed();                                    // other CTAs of the cluster read while selecting
    cluster_wait();
  }

  // move m copies the K row, the V row and the position of entry src[m] (>= B) into the hole dst[m] (< B).
  // Sources and destinations never overlap, rows are copied bit-exactly.  One warp per move.
  const long long row_bytes = static_cast<long long>(p.d) * elem_bytes;
  const int vec = static_cast<int>(row_bytes / 16);
  const long long head = static_cast<long long>(g) * p.cap;
  // (row = 2 * vec pieces of 16 bytes, K then V; a warp keeps kMovesInFlight moves in flight, since one
  // load-then-store at a time would leave the copy latency-bound)
  constexpr int kMovesInFlight = 4;
  const int wstride = Cn * (kCompressThreads / 32);
  for (int mv0 = rank * (kCompressThreads / 32) + warp; mv0 < total_holes; mv0 += wstride * kMovesInFlight) {
    int src[kMovesInFlight], dst[kMovesInFlight];
#pragma unroll
    for (int u = 0; u < kMovesInFlight; ++u) {
      const int mv = mv0 + u * wstride;
      src[u] = mv < total_holes ? msrc[mv] : -1;
      dst[u] = mv < total_holes ? mdst[mv] : -1;
    }
    for (int i = lane; i < 2 * vec; i += 32) {
      const long long off = (i < vec ? 0 : p.v_off) + static_cast<long long>(i < vec ? i : i - vec) * 16;
      uint4 val[kMovesInFlight];
#pragma unroll
      for (int u = 0; u < kMovesInFlight; ++u)
        if (src[u] >= 0) val[u] = *reinterpret_cast<const uint4*>(blob + off + (head + src[u]) * row_bytes);
#pragma unroll
      for (int u = 0; u < kMovesInFlight; ++u)
        if (src[u] >= 0) *reinterpret_cast<uint4*>(blob + off + (head + dst[u]) * row_bytes) = val[u];
    }
    if (lane < kMovesInFlight && src[0] >= 0) {
      int sj = -1, dj = -1;
#pragma unroll
      for (int u = 0; u < kMovesInFlight; ++u)
        if (lane == u) { sj = src[u]; dj = dst[u]; }
      if (sj >= 0) pos[dj] = pos[sj];
    }
  }
  __syncthreads();
  if (tid == 0) stamp_end(p);
  if (tid == 0 && sh.wait_ctl[0]) atomicExch(reinterpret_cast<int*>(ws), -4 /* KVC_ETIMEOUT */);
}

}  // namespace kvc
