// Tensor-core kernels for bf16 (sm_100a): attention (a1, Eq. 1) and score (a2, Eq. 4).
// Operands are staged in shared memory by TMA in the 128-byte-swizzled layouts tcgen05.mma reads,
// accumulators live in TMEM, and only the two dense contractions (Q K^T and P V) use the tensor
// cores; softmax, masking and the score reduction run on the CUDA cores in fp32.
#pragma once
#include <cuda.h>
#include <stddef.h>
#include "geom.cuh"
#include "ptx.cuh"

namespace kvc {

static constexpr int kSubTileBytes = 128 * 128;   // 128 rows x 64 bf16 (one 128-byte swizzled row each)

// Row packing shared by both kernels: for kv-head g the G query heads that share it are stacked
// with the tokens, row r = (token - tok0) * G + (head - g*G), so keys and values are read once per
// kv-head.  A tile holds TOK = 128 / G tokens (TOK * G <= 128 rows).


// K/V ring slots of the attention kernel, half of them for K: with one row tile per CTA the shared memory of the second Q tile
// and what is left beside it hold two more.
template <int R> __host__ __device__ constexpr int attn_stages() { return R == 1 ? 6 : 4; }

// ------------------------------------------------------------------------------------------------
// a0 + a1: append (Alg. 1) and attention (Eq. 1).  Two 128-row tiles (A, B) per CTA, software pipelined,
// with the key range optionally split over the CTAs of a thread-block cluster.  Keys are the cache rows
// [0, n_c) followed by the block's own tokens, which are read from the k/v inputs directly.
//   warps 0-3   softmax of tile A     (thread = one row = one TMEM lane), 216 registers
//   warps 4-7   softmax of tile B
//   warp  8     TMA producer: Q tiles once, then K_j and V_j through a ring of 32 KB slots, one half of it for each kind
//   warp  9     issues S_t = Q_t K_j^T (one lane), warp 10 O_t += P_t V_j.  P is handed over in two halves (64 keys each) so
//               the first PV MMAs start while the second half of the exponentials is still being computed.
//   warp  11    a0: stores the block's key / value tiles into the cache from their ring slots (TMA stores)
// The two softmax groups take turns on the exponentials (named barriers): while one tile's exponentials
// occupy the CUDA cores the other group loads its S and finds its maxima.
// TMEM columns: S [0,128)  P_A [128,192)  P_B [192,256)  O_A [256,384)  O_B [384,512).  S is not kept under P: it is free
// again as soon as a softmax group has it in registers, and the other group's next S is computed during the exponentials.
// What binds the key loop is then the way from one S to the next (cycles, with one row tile per CTA): 240 for the load, 220
// until the issuer sees all four warps past it, 630 of MMAs (Q and K both come from shared memory, 128 B a cycle), 300 - 450 until
// the warps see the result; the exponentials of an item take 1400, and TMEM has no columns for a second S.  With P over S, as it
// was before, the way was S -> maxima -> exponentials -> P V -> next S, with two row tiles in turns.  Requests before / after:
// tiled image 2670 -> 2535 us, video 8370 -> 7966, long video 11869 -> 11368, image 2731 -> 2650, proxies 1796 -> 1735; the
// results are the same bits.
// (Measured and dropped: eight softmax warps per row tile, two threads per row, also in the form where a CTA
// with a single row tile lends it the other tile's warps -- no faster; a polynomial 2^x on the FMA pipe for part
// of the columns -- slower; S in two halves of 64 keys -- an MMA with N = 64 takes as long as one with 128, long video 13250 us;
// one thread for both kinds of MMA -- four commits an item, 14540; exponentials against the running maximum with the tile's
// maximum found afterwards -- slower, the period is then bound by the two exponential phases, which that form lengthens.)
// The running output is rescaled lazily: a row keeps its reference maximum until the true maximum
// has grown by more than 2^8, so P stays below 256 and O rarely needs touching.
//
// Key split: with cluster size S the CTA of cluster rank s handles key tiles [s*T/S, (s+1)*T/S) of
// its row tile (one per CTA then) and ends with a partial (O, m, l).  The partials are exchanged through distributed
// shared memory: rank s owns rows [s*128/S, (s+1)*128/S), every CTA sends the rows of another owner, (m, l) behind
// them, in one bulk copy, and each rank combines and writes its rows.  Nothing but the final result goes to HBM.
// Row tiles per CTA: R = 2 as described, or R = 1.  A CTA with one row tile runs it twice over: softmax group t takes its
// key tiles t, t+2, ... with P, O, maximum and row sum of its own (tile B's TMEM columns), and
// the two partial results are merged at the end, column half by column half straight from TMEM.  That doubles the CTA
// count at 0.80 per row tile and key tile, against half of 1.66 in a pair.
// What bounds a launch (device stamps, us): 1.3 - 1.4 until the first S (dependency wait, TMA, MMA), then 0.80 per key tile
// with one row tile or 1.66 with two, 1.5 - 1.7 for the epilogue, about 3.5 for the combine of a key split.
// (While S lay under P, 0.94 and 1.78 a key tile: with the output through shared memory, the merge from TMEM, the six-slot ring
// and cluster barriers that order no memory, tiled image (13 key tiles, 128 CTAs) 16.4 -> 14.5, video (18 key tiles split over
// two, 112 CTAs) 17.5 -> 15.3; two row tiles (long video) 73.3 -> 73.1.)
// grid (R == 1 ? tiles * S : tiles - n_pairs, Hkv, nl) with tiles = ceil(n/TOK), cluster (S,1,1), block 384,
// dynamic smem (R + attn_stages<R>()) * (D/64) * 16 KB + 1 KB.
static constexpr int kAttnThreads = 384;

struct TcSmemAttn {
  uint64_t q_full[2], kv_full[6], kv_empty[6], s_full[2], s_free, p_half[2][2], pv_done[2];
  uint64_t mma_done[2];      // a wait ran out: every MMA that this issuer issued is complete
  uint64_t comb_full;        // key split: the other ranks' partial rows have landed in this CTA's shared memory
  uint32_t tmem_base;
  int s_issued;              // two row tiles: the last item whose S has been issued
  int wait_ctl[2];           // [0] abort flag, [1] wait limit in units of 1024 cycles (see mbar_wait)
};
static_assert(offsetof(TcSmemAttn, kv_full) == offsetof(TcSmemAttn, q_full) + 2 * sizeof(uint64_t));   // (walked as one array)

template <int D, int R>
__global__ void __launch_bounds__(kAttnThreads, 1) attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q,
                                                                   const __grid_constant__ CUtensorMap tm_k,
                                                                   const __grid_constant__ CUtensorMap tm_v,
                                                                   const __grid_constant__ CUtensorMap tm_kin,
                                                                   const __grid_constant__ CUtensorMap tm_vin,
                                                                   const __grid_constant__ CUtensorMap tm_out,
                                                                   char* __restrict__ cache,
                                                                   __nv_bfloat16* __restrict__ out,
                                                                   char* __restrict__ ws, Geom p, int S, int n_pairs) {
  constexpr int kStages = attn_stages<R>();
  constexpr int NSUB = D / 64;
  constexpr int TILE_BYTES = NSUB * kSubTileBytes;
  constexpr uint32_t TMEM_COLS = 512;
  constexpr float kRescaleThreshold = 8.f;      // log2 units
  // The turn is handed over when this quarter of P has been stored (2: tiled image 2540 -> 2560 us, video 7945 -> 7965).
  constexpr int kTellAt = 3;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;                            // R tiles; after the key loop: the output tiles
  uint8_t* ring = smem + R * TILE_BYTES;         // kStages tiles; after the key loop: the partials of a key split
  __shared__ TcSmemAttn sh;

  // Without a key split the row tiles that see the most keys, the last ones, start first, and the kv-heads take turns: in
  // a launch of several waves the short CTAs then fill the end (2048 tokens in one pass, 28 / 4 heads, 4 layers with five
  // short blocks behind it: 316 -> 241 us), and in one wave the longest CTAs are not the last to get an SM (requests: tiled
  // image 2735 -> 2661 us, hybrid long video 3144 -> 3108, long video no difference).
  const int lin = blockIdx.y * gridDim.x + blockIdx.x;
  const bool ordered = S == 1;
  const int layer = blockIdx.z, g = ordered ? lin % gridDim.y : blockIdx.y;
  const int bx = ordered ? gridDim.x - 1 - lin / gridDim.y : blockIdx.x;
  const int split = S > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  // R = 1: a row tile per CTA (or per cluster).  R = 2: the first n_pairs CTAs of a kv-head take two row tiles each, the
  // others one of the rest.
  const int TOK = 128 / p.G, rows = TOK * p.G;
  const bool has_B = R == 2 && bx < n_pairs;
  const int tile0 = R == 1 ? bx / S : has_B ? 2 * bx : n_pairs + bx;
  const int tokA = tile0 * TOK, tokB = tokA + TOK, tok_end = has_B ? tokB + TOK : tokB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int last_tok = min(tok_end, p.n) - 1;
  // Key tiles this pair of row tiles can see: Tc tiles of the cache (rows [0, n_c), the last one possibly
  // partial), then the block's own keys in tiles of 128 tokens, read straight from the k/v inputs.
  const int Tc = (p.n_c + 127) / 128;
  const int T = Tc + (last_tok + 128) / 128;
  const int t_begin = split * T / S, t_end = (split + 1) * T / S;
  const int Tl = t_end - t_begin;                // key tiles of this CTA (0 is possible when S > T)
  // A CTA with one row tile runs it twice over: softmax group t takes the key tiles t, t+2, ... with accumulators, maxima and sums
  // of their own (the TMEM columns of tile B are free), two key tiles are in flight as with two row tiles, and the two partial
  // results are merged at the end.  (With Tl = 1 group 1 has none; Tl = 0 happens with a key split, for the first rows of a block
  // that see less of it than the last ones.)
  const bool alt = !has_B;
  const int n_it0 = alt ? (Tl + 1) / 2 : Tl, n_it1 = alt ? Tl / 2 : Tl;   // key tiles of group 0 / 1

  // block tiles [u_lo, u_hi) of this CTA that it appends to the cache (see warp 11): those that begin in its rows
  const int u_lo = max(max(t_begin - Tc, 0), (tokA + 127) / 128), u_hi = min(t_end - Tc, (tok_end + 127) / 128);
  const bool appends = u_hi > u_lo;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.q_full[i], 1); mbar_init(&sh.s_full[i], 1); mbar_init(&sh.pv_done[i], 1);
      mbar_init(&sh.p_half[i][0], 4); mbar_init(&sh.p_half[i][1], 4);     // one arrival per softmax warp
    }
    mbar_init(&sh.s_free, 4);                                             // (likewise)
    for (int i = 0; i < kStages; ++i) { mbar_init(&sh.kv_full[i], 1); mbar_init(&sh.kv_empty[i], appends ? 2 : 1); }
    sh.s_issued = -1;
    sh.wait_ctl[0] = 0; sh.wait_ctl[1] = p.wait_limit_k;
    mbar_init(&sh.mma_done[0], 1); mbar_init(&sh.mma_done[1], 1);
    mbar_init(&sh.comb_full, 1);
    // key split: every other rank of the cluster will copy its partial of this rank's rows here
    if (S > 1) mbar_expect_tx(&sh.comb_full, (S - 1) * (128 / S) * (D + 4) * 4);
    mbar_fence_init();
  }
  // rows of the Q tiles that TMA never writes (rows >= TOK*G) must still be finite
  {
    const int pad16 = (128 - rows) * 8;          // 16-byte units per sub-tile
    for (int i = threadIdx.x; i < R * NSUB * pad16; i += blockDim.x) {
      const int sub = i / pad16, rem = i % pad16;
      reinterpret_cast<uint4*>(sQ + sub * kSubTileBytes + rows * 128)[rem] = make_uint4(0, 0, 0, 0);
    }
  }
  fence_proxy_async_smem();
  if (warp == 8) {
    tmem_alloc(&sh.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sh.tmem_base;
  volatile int* abort_flag = sh.wait_ctl;

  // The items of this CTA, in the order in which everything below takes them: item i is softmax group i & 1's next key tile.
  // Two row tiles: items 2j and 2j + 1 are key tile j of row tile A and B; one row tile: item i is key tile i.
  const int n_items = has_B ? 2 * Tl : Tl;

  if (warp >= 8) {
    reg_dec<56>();                               // (with 64 or 72 the compiler spills in the softmax groups of some forms: 2 - 8 % slower)
    // Ring: K tiles go round the first kSlots slots, V tiles round the others.
    constexpr int kSlots = kStages / 2;
    uint32_t loads = ~3u;                          // per barrier, q_full and kv_full: the parity of the last phase that loads complete
    auto load_tile = [&](int j, int v) {           // K (v = 0) or V (1) of local key tile j; false: gave up
      const int slot = v * kSlots + j % kSlots, round = j / kSlots, kt = t_begin + j;
      if (round > 0 && !mbar_wait(&sh.kv_empty[slot], (round - 1) & 1, abort_flag)) return false;
      mbar_expect_tx(&sh.kv_full[slot], TILE_BYTES);
      loads ^= 4u << slot;
      uint8_t* dst = ring + slot * TILE_BYTES;
      if (kt < Tc) {                             // cache rows kt*128 .. (rows past n_c are masked by the softmax)
        for (int sub = 0; sub < NSUB; ++sub) tma_load_4d(dst + sub * kSubTileBytes, v ? &tm_v : &tm_k, &sh.kv_full[slot], sub * 64, kt * 128, g, layer);
      } else {                                   // block tokens (kt - Tc)*128 .. (tokens past n are zero-filled)
        for (int sub = 0; sub < NSUB; ++sub) tma_load_4d(dst + sub * kSubTileBytes, v ? &tm_vin : &tm_kin, &sh.kv_full[slot], sub * 64, g, (kt - Tc) * 128, layer);
      }
      return true;
    };
    if (warp == 8) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0) {
        tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v);
        tma_prefetch_desc(&tm_kin); tma_prefetch_desc(&tm_vin); tma_prefetch_desc(&tm_out);
      }
      // While the previous kernel drains: ask L2 for the Q tiles and the first two key / value tiles (a hint only,
      // nothing is read into the SM before the wait below), so that the first loads find them there.
      if (Tl > 0 && lane < 2 + 2 * NSUB * min(Tl, 2)) {
        if (lane < 2) {
          if (lane == 0 || has_B)
            for (int sub = 0; sub < NSUB; ++sub) tma_prefetch_l2_4d(&tm_q, sub * 64, g * p.G, lane ? tokB : tokA, layer);
        } else {
          const int i = (lane - 2) / NSUB, sub = (lane - 2) % NSUB;      // K or V of key tile t_begin + i/2
          const int kt = t_begin + (i >> 1);
          if (kt < Tc) tma_prefetch_l2_4d((i & 1) ? &tm_v : &tm_k, sub * 64, kt * 128, g, layer);
          else tma_prefetch_l2_4d((i & 1) ? &tm_vin : &tm_kin, sub * 64, g, (kt - Tc) * 128, layer);
        }
      }
      __syncwarp();
      if (lane == 0) {
        pdl_wait();                                // the previous block's compaction is done with the cache
        if (p.early) pdl_launch_dependents();
        stamp_begin(p);
      }
      if (lane == 0 && Tl > 0) {
        mbar_expect_tx(&sh.q_full[0], NSUB * rows * 128);
        for (int sub = 0; sub < NSUB; ++sub)
          tma_load_4d(sQ + sub * kSubTileBytes, &tm_q, &sh.q_full[0], sub * 64, g * p.G, tokA, layer);
        // In the order in which they are needed: an SM takes in 64 bytes a cycle, and V tiles asked for beside the first K tile
        // hold it up (three key tiles: 0.5 us of a call of 8).  Behind the first fill K runs a tile ahead of V, as S does.
        const int fill = min(Tl, kSlots);
        for (int j = 0; j < fill; ++j) {
          load_tile(j, 0);
          if (j == 0 && has_B) {                   // (row tile A can start on Q_A and the first K tile)
            mbar_expect_tx(&sh.q_full[1], NSUB * rows * 128);
            for (int sub = 0; sub < NSUB; ++sub)
              tma_load_4d(sQ + TILE_BYTES + sub * kSubTileBytes, &tm_q, &sh.q_full[1], sub * 64, g * p.G, tokB, layer);
          }
          load_tile(j, 1);
        }
        for (int j = fill; j < Tl + 1; ++j) {
          if (j < Tl && !load_tile(j, 0)) break;
          if (j > fill && !load_tile(j - 1, 1)) break;
        }
        // The block keeps its shared memory until they have landed, whoever has given up waiting for them.  (Barriers without a
        // load are in their first phase, and the one before counts as complete.  Requests: no difference beyond their spread.)
        if (!has_B) loads |= 2u;
#pragma unroll 1
        for (int i = 0; i < 2 + kStages; ++i) mbar_drain(&sh.q_full[0] + i, loads >> i & 1);
      }
    } else if (warp == 11) {
      // ---------------------------------------------------------------- a0 append (Alg. 1: C <- C u (K_i, V_i))
      // The block's keys and values pass through the ring as key tiles anyway: such a tile is stored from its ring slot into
      // cache rows n_c + 128u .. with one TMA store per 64 columns (rows past the block are zero in the tile and land in unused
      // cache rows or are clipped at cap).  Among the CTAs that load block tile u, the one whose rows contain token 128u owns
      // it.  Nobody in this kernel reads the appended rows.  In a CTA that owns tiles every slot is handed back by this warp,
      // too, once a store has read it.
      if (appends) {
        pdl_wait();                                // the previous block's compaction is done with the cache
        int* pos = reinterpret_cast<int*>(cache + layer * p.cache_ls + p.pos_off) + static_cast<long long>(g) * p.cap + p.n_c;
        for (int u = u_lo; u < u_hi; ++u)
          for (int i = u * 128 + lane; i < min(p.n, u * 128 + 128); i += 32) pos[i] = static_cast<int>(p.pos0 + i);
        if (lane == 0) {
          for (int i = 0; i < 2 * Tl; ++i) {       // K and V of local key tile i / 2
            const int j = i >> 1, slot = (i & 1) * kSlots + j % kSlots, u = t_begin + j - Tc;
            if (!mbar_wait(&sh.kv_full[slot], (j / kSlots) & 1, abort_flag)) break;
            if (u >= u_lo && u < u_hi) {
              for (int sub = 0; sub < NSUB; ++sub)
                tma_store_4d((i & 1) ? &tm_v : &tm_k, ring + slot * TILE_BYTES + sub * kSubTileBytes, sub * 64, p.n_c + u * 128, g, layer);
              tma_store_commit();
              tma_store_wait_read();
            }
            mbar_arrive(&sh.kv_empty[slot]);
          }
        }
      }
    } else if (warp == 9) {
      // ---------------------------------------------------------------- issuer of S = Q K^T, item by item
      // S has one buffer of 128 columns: the next item's S is issued as soon as a group has this one in its registers, and is
      // there by the time the other group comes for it.  (One thread for both kinds of MMA is too slow: four commits an item.)
      if (lane == 0 && n_items > 0) {
        constexpr uint32_t idesc_qk = idesc_bf16_f32(128, 128, 0, 0);
        constexpr uint32_t hi = smem_desc_hi_sw128(1024);
        const uint32_t q_lo0 = smem_desc_lo(smem_u32(sQ), 16), k_lo0 = smem_desc_lo(smem_u32(ring), 16);   // K-major operands
        bool ok = mbar_wait(&sh.q_full[0], 0, abort_flag);
        for (int i = 0; i < n_items && ok; ++i) {
          const int t = i & 1, j = has_B ? i >> 1 : i, slot = j % kSlots;
          if (!has_B || t == 0) ok = mbar_wait(&sh.kv_full[slot], (j / kSlots) & 1, abort_flag);
          if (ok && has_B && i == 1) ok = mbar_wait(&sh.q_full[1], 0, abort_flag);
          if (ok && i > 0) ok = mbar_wait_spin(&sh.s_free, (i - 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t q_lo = q_lo0 + (has_B ? t : 0) * (TILE_BYTES >> 4), k_lo = k_lo0 + slot * (TILE_BYTES >> 4);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {      // 16 of the d columns per MMA
            const uint32_t off = ((kk / 4) * kSubTileBytes + (kk % 4) * 32) >> 4;
            mma_ss_lh(tmem, q_lo + off, hi, k_lo + off, hi, idesc_qk, kk > 0);
          }
          mma_commit(&sh.s_full[t]);
          if (has_B) *static_cast<volatile int*>(&sh.s_issued) = i;
          if (!has_B || t == 1) mma_commit(&sh.kv_empty[slot]);
        }
      }
    } else {
      // ---------------------------------------------------------------- issuer of O_t += P_t V, item by item, half by half
      // With two row tiles per CTA it lets the S of the item after next go first: that one is wanted soon, while P V of this
      // item has time until the group's next P (long video 11675 -> 11457 us per request, hybrid 3083 -> 3049; with one row
      // tile per CTA 1 % slower).
      if (lane == 0 && n_items > 0) {
        constexpr uint32_t idesc_pv = idesc_bf16_f32(128, D, 0, 1);
        constexpr uint32_t hi = smem_desc_hi_sw128(1024);
        const uint32_t v_lo0 = smem_desc_lo(smem_u32(ring) + kSlots * TILE_BYTES, kSubTileBytes);   // MN-major operand
        bool ok = true;
        for (int i = 0; i < n_items && ok; ++i) {
          const int t = i & 1, it = i >> 1, j = has_B ? it : i, slot = j % kSlots;
          if (!has_B || t == 0) ok = mbar_wait(&sh.kv_full[kSlots + slot], (j / kSlots) & 1, abort_flag);
          const uint32_t v_lo = v_lo0 + slot * (TILE_BYTES >> 4), tP = tmem + 128 + t * 64, tO = tmem + 256 + t * 128;
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            ok = ok && mbar_wait_spin(&sh.p_half[t][half], it & 1, abort_flag);
            if (has_B && half == 0) ok = ok && word_wait_spin(&sh.s_issued, min(i + 2, n_items - 1), abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
#pragma unroll
            for (int kk = 4 * half; kk < 4 * half + 4; ++kk)   // 16 keys per MMA, 64 keys per half
              mma_ts_lh(tO, tP + kk * 8, v_lo + kk * (2048 >> 4), hi, idesc_pv, it > 0 || kk > 0);
          }
          if (!ok) break;
          mma_commit(&sh.pv_done[t]);
          if (!has_B || t == 1) mma_commit(&sh.kv_empty[kSlots + slot]);
        }
      }
    }
    __syncwarp();
    // One row tile: the epilogue writes over the ring and the Q tile once both key chains are complete, which says
    // nothing about the stores above; warp 11 tells it here that no store reads the ring any more.
    if (alt && warp == 11) named_barrier_arrive(5, 256 + 32);
    if (S > 1) { cluster_arrive_relaxed(); cluster_wait(); }  // the cluster barriers of the combine below
    // No barrier of the whole block at the end: TMEM is given back as soon as the softmax warps have read it for the last time,
    // and every warp leaves when it is done (requests: video 7944 -> 7855 us, query-agnostic 1268 -> 1261, image 2652 -> 2643).
    // The softmax warps may be here without their results, when a wait ran out.  Then an issuer can have MMAs under way, or a
    // tile can have landed for it that it issued some on: it comes here behind its loop and sees them to their end.
    // (The price is the room of this code among the other: image 2627 -> 2643 us, video 7852 -> 7864, tiled image and image from a
    // graph within their spread.  With a flag of its own, so that warp 8 need not come behind the issuers: video 7935.)
    if (warp == 9 || warp == 10) {
      named_barrier(6, 256 + 64);
      if (__builtin_expect(abort_flag[0] != 0, 0) && lane == 0) {
        mma_commit(&sh.mma_done[warp - 9]);
        mbar_drain(&sh.mma_done[warp - 9], 0);
      }
      __syncwarp();
      named_barrier_arrive(7, 96);
    }
    if (warp == 8) {
      named_barrier(7, 96);
      tc_fence_after_sync();
      tmem_dealloc(tmem, TMEM_COLS);
    }
    if (S > 1) { cluster_arrive_relaxed(); cluster_wait(); }
    if (lane == 0) tma_store_wait_all();        // the appended rows are in the cache before the kernel ends
  } else {
    reg_inc<216>();
    // ---------------------------------------------------------------- softmax + epilogue of tile t
    const int t = warp >> 2;
    const int r = (warp & 3) * 32 + lane;                     // row of the tile = TMEM lane
    const int tok0 = (t && !alt) ? tokB : tokA;             // (both groups hold the rows of tile A when they alternate)
    const int tok = tok0 + r / p.G, hh = r % p.G;
    const bool row_valid = r < rows && tok < p.n;
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tmem_S = tmem + lane_addr, tmem_P = tmem + 128 + t * 64 + lane_addr, tmem_O = tmem + 256 + t * 128 + lane_addr;
    float m_ref = -INFINITY, l = 0.f;                        // reference maximum (log2 units) and row sum
    bool ok = true;
    const int first = alt ? t : 0, step = alt ? 2 : 1;       // local key tiles of this group: first, first + step, ...
    // Turn taking (named barrier 2 + t = "group t may go", 128 waiters + 128 arrivals).  Group 0 goes first.
    const bool turns = Tl > 0;
    if (turns && t == 1) named_barrier_arrive(2, 256);
    {
      for (int jj = first, it = 0; jj < Tl; jj += step, ++it) {
        const int kt = t_begin + jj;                          // key tile index
        // Waits that gave up only skip the arithmetic: the turn barrier is passed on every path, once per key
        // tile and warp, so the other row tile never waits for a turn that is not handed over.
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&sh.s_full[t], it & 1, abort_flag));
        bool took_turn = false, told = false;
        const bool hand_over = t == 0 ? it < n_it1 : it + 1 < n_it0;   // the other group has a key tile left: its it-th (group 0 asks) or (it+1)-th
        if (ok) do {
        tc_fence_after_sync();
        uint32_t sr[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tmem_S + c * 32, sr + c * 32);
        // O_t holds every earlier tile, and the columns of P are free?  (asked while S is on its way; long so as a rule)
        const bool pv_ready = it > 0 && mbar_test_wait(&sh.pv_done[t], (it - 1) & 1);
        tmem_wait_ld();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.s_free);               // the other group's next S may be computed
        // columns [0, lim) of this tile are visible: a cache tile ends at row n_c, a block tile at the row's
        // own token (causal inside the block); only the last cache tile and diagonal tiles need the mask
        const int u = kt - Tc;                                // >= 0: tile of the block's own tokens
        const int lim = u < 0 ? p.n_c - kt * 128 : tok + 1 - u * 128;
        if (__builtin_expect(u < 0 ? lim < 128 : (u + 1) * 128 > tok0 + 1, 0)) {
          if constexpr (R == 1) {
            // As bits of a word per quarter: a predicate comes from each with less code than from a comparison (requests, with
            // the two unlikely branches told so: image 2639 -> 2627 us, image from a graph 1499 -> 1480, tiled image 2535 ->
            // 2524, video 7856 -> 7831, query-agnostic 1263 -> 1256; nothing with two row tiles).
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int left = lim - 32 * c;                  // visible columns from this quarter on
              const uint32_t see = left >= 32 ? 0xffffffffu : left <= 0 ? 0u : (1u << left) - 1u;
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (!(see >> i & 1u)) sr[c * 32 + i] = 0xff800000u;   // -inf
            }
          } else {
#pragma unroll
            for (int c = 0; c < 128; ++c)
              if (c >= lim) sr[c] = 0xff800000u;              // -inf
          }
        }
        float mx4[8];                                         // independent chains of three-input maxima
#pragma unroll
        for (int i = 0; i < 8; ++i) mx4[i] = fmaxf(__uint_as_float(sr[i]), __uint_as_float(sr[8 + i]));
#pragma unroll
        for (int c = 16; c < 128; c += 16) {
#pragma unroll
          for (int i = 0; i < 8; ++i) mx4[i] = fmax3(mx4[i], __uint_as_float(sr[c + i]), __uint_as_float(sr[c + 8 + i]));
        }
        const float mx = fmaxf(fmax3(mx4[0], mx4[1], mx4[2]), fmaxf(fmax3(mx4[3], mx4[4], mx4[5]), fmaxf(mx4[6], mx4[7])));
        const float m_new = mx * p.scale_log2;                // scale > 0
        const bool grow = m_new > m_ref + kRescaleThreshold;  // (first tile: m_ref is -infinity)
        if (__builtin_expect(__any_sync(0xffffffffu, grow || !pv_ready), 0)) {
          if (it == 0) {
            m_ref = m_new == -INFINITY ? 0.f : m_new;
          } else {
            ok = __all_sync(0xffffffffu, mbar_wait(&sh.pv_done[t], (it - 1) & 1, abort_flag));
            if (!ok) break;
            if (__any_sync(0xffffffffu, grow)) {
              tc_fence_after_sync();
              const float f = grow ? fast_exp2(m_ref - m_new) : 1.f;
              if (grow) { m_ref = m_new; l *= f; }
#pragma unroll
              for (int c = 0; c < D / 32; ++c) {
                uint32_t o[32];
                tmem_ld32(tmem_O + c * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                tmem_st32(tmem_O + c * 32, o);
              }
            }
          }
        }
        tc_fence_after_sync();
        // Only the exponentials are taken in turns: loading S and finding the row maxima overlap the other
        // tile's exponentials.
        if (turns) { named_barrier(2 + t, 256); took_turn = true; }
        // (packed fp32: one instruction scales two columns, one adds two exponentials to the partial sums)
        const uint64_t scale2 = f32x2(p.scale_log2, p.scale_log2), neg_m2 = f32x2(-m_ref, -m_ref);
        uint64_t ps2[2] = {f32x2(0.f, 0.f), f32x2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float x0, x1;
            f32x2_split(fma_f32x2(f32x2(__uint_as_float(sr[c * 32 + 2 * i]), __uint_as_float(sr[c * 32 + 2 * i + 1])), scale2, neg_m2), x0, x1);
            const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
            ps2[i & 1] = add_f32x2(ps2[i & 1], f32x2(p0, p1));
            pk[i] = pack_bf16x2(p0, p1);
          }
          if (c == 2) {                                       // the first 64 keys of P have landed: the MMA warp may take them
            tmem_wait_st();
            tc_fence_before_sync();
            // one arrival per warp: 128 arrivals on one shared-memory word are served one after the other, and the
            // issuer saw the barrier complete some 300 cycles after the first of them (in-kernel stamps)
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.p_half[t][0]);
          }
          tmem_st16(tmem_P + c * 16, pk);
          if (c == kTellAt) { if (turns && hand_over) named_barrier_arrive(3 - t, 256); told = true; }
        }
        {
          float ps[4];
          f32x2_split(ps2[0], ps[0], ps[1]);
          f32x2_split(ps2[1], ps[2], ps[3]);
          l += (ps[0] + ps[1]) + (ps[2] + ps[3]);
        }
        tmem_wait_st();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.p_half[t][1]);
        } while (0);
        if (turns && !took_turn) named_barrier(2 + t, 256);   // a wait gave up before the turn was taken: take it now
        if (turns && !told && hand_over) named_barrier_arrive(3 - t, 256);
      }
      // The key loop is over: the next kernel of the stream may be scheduled and set itself up while this one
      // writes its results.  (Triggered at the start instead, the waiting CTAs of the next attention launch take the
      // SMs that the compress kernel of the previous layer, ready on a side stream, could use.)
      if (threadIdx.x == 0) pdl_launch_dependents();
    }
    // ---- epilogue.  With two row tiles per CTA output rows leave through shared memory and TMA: a thread holds one row,
    // and 32 threads storing 16 bytes each of 32 different rows cost a sector per thread and instruction.
    const long long head_row = static_cast<long long>(g) * p.G;       // output / lse row of (token, hh): token * Hq + head_row + hh
    auto out_chunk = [&](int tile, int c16) -> uint4* {               // 16-byte piece c16 of row r in the swizzled output tile
      return reinterpret_cast<uint4*>(sQ + tile * TILE_BYTES + (c16 >> 3) * kSubTileBytes + r * 128 + (((c16 & 7) ^ (r & 7)) << 4));
    };
    // the last read of TMEM is done: it may be given back
    auto tmem_done = [&]() { tc_fence_before_sync(); named_barrier_arrive(6, 256 + 64); };
    if (has_B) {
      // Two row tiles: a group owns its rows.  Normalise, round, store the tile over its Q tile and let TMA write it out (tokens
      // past n are clipped).  Nothing reads that Q tile any more: this group has had its last S (s_full), which is what its last P
      // was made from, and only the S of its own row tile are made from it.
      ok = ok && mbar_wait(&sh.pv_done[t], (Tl - 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);                       // the TMEM accesses below are warp-wide
      if (ok) {
        tc_fence_after_sync();
        const float inv = 1.f / l;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(tmem_O + c * 32, o);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint4 vv;
            vv.x = pack_bf16x2(__uint_as_float(o[8 * i + 0]) * inv, __uint_as_float(o[8 * i + 1]) * inv);
            vv.y = pack_bf16x2(__uint_as_float(o[8 * i + 2]) * inv, __uint_as_float(o[8 * i + 3]) * inv);
            vv.z = pack_bf16x2(__uint_as_float(o[8 * i + 4]) * inv, __uint_as_float(o[8 * i + 5]) * inv);
            vv.w = pack_bf16x2(__uint_as_float(o[8 * i + 6]) * inv, __uint_as_float(o[8 * i + 7]) * inv);
            *out_chunk(t, c * 4 + i) = vv;
          }
        }
        if (row_valid) {
          float* lse = reinterpret_cast<float*>(ws_slot(ws, p, layer) + p.lse_off);
          lse[static_cast<long long>(tok) * p.Hq + head_row + hh] = (m_ref + log2f(l)) * 0.6931471805599453f;
        }
        fence_proxy_async_smem();
      }
      tmem_done();
      named_barrier(1 + 3 * t, 128);                           // (ids 1 and 4)
      if (r == 0 && ok) {
        for (int sub = 0; sub < NSUB; ++sub)
          tma_store_4d(&tm_out, sQ + t * TILE_BYTES + sub * kSubTileBytes, sub * 64, g * p.G, tok0, layer);
        tma_store_commit();
        tma_store_wait_read();
      }
    } else {
      // One row tile, two key chains.  Both accumulators sit in TMEM on the same lanes, so no thread has to hand rows
      // over: group t takes half the columns of both, and only (m, l) are exchanged (through the TMEM columns of P).
      constexpr int H = D / 2;
      if (ok && n_it0 > 0) ok = mbar_wait(&sh.pv_done[0], (n_it0 - 1) & 1, abort_flag);
      if (ok && n_it1 > 0) ok = mbar_wait(&sh.pv_done[1], (n_it1 - 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc_fence_after_sync();
        tmem_st2(tmem_P, __float_as_uint(l > 0.f ? m_ref : -INFINITY), __float_as_uint(l));   // -inf: no key of the row seen
        tmem_wait_st();
        tc_fence_before_sync();
      }
      named_barrier(5, 256 + 32);                              // both groups are here, and no store reads the ring
      // This CTA's shared memory may be written by the cluster: everything that used it is complete and nothing was
      // written there through the generic proxy, so the arrival need not order memory (a release costs 0.4 us here).
      if (S > 1) cluster_arrive_relaxed();
      float m_all = -INFINITY, L = 0.f, w0 = 0.f, w1 = 0.f;
      if (ok) {
        tc_fence_after_sync();
        uint32_t mb, lb;
        tmem_ld2(tmem + 128 + (1 - t) * 64 + lane_addr, mb, lb);
        tmem_wait_ld();
        const float m_own = l > 0.f ? m_ref : -INFINITY, m_oth = __uint_as_float(mb), l_oth = __uint_as_float(lb);
        m_all = fmaxf(m_own, m_oth);
        const float w_own = m_own == -INFINITY ? 0.f : fast_exp2(m_own - m_all);
        const float w_oth = m_oth == -INFINITY ? 0.f : fast_exp2(m_oth - m_all);
        L = fmaf(w_oth, l_oth, w_own * l);
        w0 = t == 0 ? w_own : w_oth;
        w1 = t == 0 ? w_oth : w_own;
      }
      const uint32_t tO0 = tmem + 256 + lane_addr + t * H, tO1 = tO0 + 128;    // this group's columns of both chains' O
      const bool both = n_it1 > 0;                             // (one key tile: chain 1 has no O)
      if (R == 2 || S == 1) {                                  // (a key split always has one row tile per CTA)
        if (ok) {
          const float inv = 1.f / L, a0 = w0 * inv, a1 = w1 * inv;
#pragma unroll
          for (int c = 0; c < H / 32; ++c) {
            uint32_t o[32], q[32];
            tmem_ld32(tO0 + c * 32, o);
            if (both) tmem_ld32(tO1 + c * 32, q);
            tmem_wait_ld();
            float f[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) f[i] = both ? fmaf(a1, __uint_as_float(q[i]), a0 * __uint_as_float(o[i])) : a0 * __uint_as_float(o[i]);
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = pack_bf16x2(f[2 * i], f[2 * i + 1]);
            if constexpr (R == 1) {
              // Straight from the registers, a sector per store: no barrier, no wait for a copy to leave (requests: image
              // 2897 -> 2842 us, image from a graph 1552 -> 1514, tiled image 2831 -> 2736).
              if (row_valid) {
                __nv_bfloat16* dst = out + layer * p.out_ls + (static_cast<long long>(tok) * p.Hq + head_row + hh) * D + t * H + c * 32;
                if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
                  st_global_v8(dst, pk);
                  st_global_v8(dst + 16, pk + 8);
                } else {
#pragma unroll
                  for (int i = 0; i < 4; ++i) reinterpret_cast<uint4*>(dst)[i] = make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
                }
              }
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) *out_chunk(0, t * (H / 8) + c * 4 + i) = make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
            }
          }
          if (row_valid && t == 0) {
            float* lse = reinterpret_cast<float*>(ws_slot(ws, p, layer) + p.lse_off);
            lse[static_cast<long long>(tok) * p.Hq + head_row + hh] = (m_all + log2f(L)) * 0.6931471805599453f;
          }
          if (R == 2) fence_proxy_async_smem();
        }
        tmem_done();
        if constexpr (R == 2) {
          named_barrier(1, 256);
          if (threadIdx.x == 0 && ok) {
            for (int sub = 0; sub < NSUB; ++sub)
              tma_store_4d(&tm_out, sQ + sub * kSubTileBytes, sub * 64, g * p.G, tok0, layer);
            tma_store_commit();
            tma_store_wait_read();
          }
        }
      } else if constexpr (R == 1) {
        // Combine the partials of the cluster (S is a power of two; rank s owns rows [s*rows_per, (s+1)*rows_per)).
        // A thread has its row's merged columns in registers.  The owner's threads keep them (up to S = 4; clusters of two
        // 15.6 -> 15.0 us, 16.6 -> 15.9; with eight 12.5 -> 13.0, hence not there); the others write theirs into
        // a staging tile whose rows carry (m, l) behind the D values, the rows of every other owner leave in ONE bulk copy
        // each (shared memory to the owner's shared memory, completing on a barrier of the owner: this GPU's memory, no
        // multicast), and the owner's threads fold in what arrived and write:
        //   O = sum_s 2^(m_s - m*) O_s / sum_s 2^(m_s - m*) l_s.
        // Over the ring: the received rows [S - 1 sources][rows_per][D + 4] and the staging tile [128][D + 4] (a row
        // stride of D + 4 floats keeps thread-per-row accesses off each other's banks).
        constexpr int RS = D + 4;
        const int rows_per = 128 / S;
        float* recv = reinterpret_cast<float*>(ring);
        float* stg = recv + (128 - rows_per) * RS;
        const bool own = S < 8 && r / rows_per == split;
        float f[H];
#pragma unroll
        for (int c = 0; c < H / 32; ++c) {
          uint32_t o[32], q[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) { o[i] = 0u; q[i] = 0u; }   // (a chain without key tiles leaves its O columns unset)
          if (ok && n_it0 > 0) tmem_ld32(tO0 + c * 32, o);
          if (ok && both) tmem_ld32(tO1 + c * 32, q);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) f[c * 32 + i] = fmaf(w1, __uint_as_float(q[i]), w0 * __uint_as_float(o[i]));
        }
        tmem_done();
        if (!own) {
#pragma unroll
          for (int k = 0; k < H / 4; ++k)
            *reinterpret_cast<float4*>(stg + r * RS + t * H + k * 4) = make_float4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
          if (t == 0) *reinterpret_cast<float2*>(stg + r * RS + D) = make_float2(m_all, L);
        }
        fence_proxy_async_smem();                              // the rows just written are read by bulk copies
        named_barrier(1, 256);
        cluster_wait();                                        // every CTA of the cluster is done with its ring
        if (threadIdx.x == 0) {
          for (int owner = 0; owner < S; ++owner) {
            if (owner == split) continue;
            const int slot = split < owner ? split : split - 1;   // this rank among the owner's other ranks
            bulk_copy_to_cluster(dsmem_addr(smem_u32(recv + slot * rows_per * RS), owner), smem_u32(stg + owner * rows_per * RS),
                                 rows_per * RS * 4, dsmem_addr(smem_u32(&sh.comb_full), owner));
          }
        }
        // The other ranks' rows have landed.  They are sent whoever has given up, so they are waited for in any case: this CTA's
        // shared memory must not go while they are on their way.
        if (__builtin_expect(!mbar_wait(&sh.comb_full, 0, abort_flag), 0)) mbar_drain(&sh.comb_full, 0);
        if (S == 8) {
          // (16 rows per owner: two warps with a row per thread would be alone; every thread takes a piece of a row)
          constexpr int CW = 16;                                 // columns per work item: (row, piece)
          const int r0 = split * rows_per;
#pragma unroll 1
          for (int item = threadIdx.x; item < rows_per * (D / CW); item += 256) {
            const int lr = item & (rows_per - 1), pc = item / rows_per, rr = r0 + lr;
            const int tk = tokA + rr / p.G;
            if (!(rr < rows && tk < p.n)) continue;
            const float* own = stg + rr * RS;
            const float* got = recv + lr * RS;                   // + source * rows_per * RS
            float m_row = own[D];
#pragma unroll 1
            for (int s2 = 0; s2 < S - 1; ++s2) m_row = fmaxf(m_row, got[s2 * rows_per * RS + D]);
            float L_row = 0.f, acc[CW];
#pragma unroll
            for (int i = 0; i < CW; ++i) acc[i] = 0.f;
#pragma unroll 1
            for (int s2 = 0; s2 < S; ++s2) {                     // (source S - 1 of the loop: this rank itself)
              const float* row = s2 < S - 1 ? got + s2 * rows_per * RS : own;
              const float2 ml = *reinterpret_cast<const float2*>(row + D);
              const float wt = ml.x == -INFINITY ? 0.f : fast_exp2(ml.x - m_row);   // -inf: the source saw no key of the row
              L_row = fmaf(wt, ml.y, L_row);
#pragma unroll
              for (int k = 0; k < CW / 4; ++k) {
                const float4 v4 = *reinterpret_cast<const float4*>(row + pc * CW + k * 4);
                acc[4 * k + 0] = fmaf(wt, v4.x, acc[4 * k + 0]); acc[4 * k + 1] = fmaf(wt, v4.y, acc[4 * k + 1]);
                acc[4 * k + 2] = fmaf(wt, v4.z, acc[4 * k + 2]); acc[4 * k + 3] = fmaf(wt, v4.w, acc[4 * k + 3]);
              }
            }
            const float inv = 1.f / L_row;
            const long long orow = static_cast<long long>(tk) * p.Hq + head_row + rr % p.G;
#pragma unroll
            for (int k = 0; k < CW / 8; ++k) {
              uint4 vv;
              vv.x = pack_bf16x2(acc[8 * k + 0] * inv, acc[8 * k + 1] * inv);
              vv.y = pack_bf16x2(acc[8 * k + 2] * inv, acc[8 * k + 3] * inv);
              vv.z = pack_bf16x2(acc[8 * k + 4] * inv, acc[8 * k + 5] * inv);
              vv.w = pack_bf16x2(acc[8 * k + 6] * inv, acc[8 * k + 7] * inv);
              reinterpret_cast<uint4*>(out + layer * p.out_ls + orow * D + pc * CW)[k] = vv;
            }
            if (pc == 0) reinterpret_cast<float*>(ws_slot(ws, p, layer) + p.lse_off)[orow] = (m_row + log2f(L_row)) * 0.6931471805599453f;
          }
        } else if (own && row_valid) {
          const float* got = recv + (r - split * rows_per) * RS;   // + source * rows_per * RS
          float m_row = m_all;
#pragma unroll 1
          for (int s2 = 0; s2 < S - 1; ++s2) m_row = fmaxf(m_row, got[s2 * rows_per * RS + D]);
          const float wt0 = m_all == -INFINITY ? 0.f : fast_exp2(m_all - m_row);   // -inf: this rank saw no key of the row
          float L_row = wt0 * L;
#pragma unroll
          for (int i = 0; i < H; ++i) f[i] *= wt0;
#pragma unroll 1
          for (int s2 = 0; s2 < S - 1; ++s2) {
            const float* row = got + s2 * rows_per * RS;
            const float2 ml = *reinterpret_cast<const float2*>(row + D);
            const float wt = ml.x == -INFINITY ? 0.f : fast_exp2(ml.x - m_row);
            L_row = fmaf(wt, ml.y, L_row);
#pragma unroll
            for (int k = 0; k < H / 4; ++k) {
              const float4 v4 = *reinterpret_cast<const float4*>(row + t * H + k * 4);
              f[4 * k + 0] = fmaf(wt, v4.x, f[4 * k + 0]); f[4 * k + 1] = fmaf(wt, v4.y, f[4 * k + 1]);
              f[4 * k + 2] = fmaf(wt, v4.z, f[4 * k + 2]); f[4 * k + 3] = fmaf(wt, v4.w, f[4 * k + 3]);
            }
          }
          const float inv = 1.f / L_row;
          const long long orow = static_cast<long long>(tok) * p.Hq + head_row + hh;
          __nv_bfloat16* dst = out + layer * p.out_ls + orow * D + t * H;
#pragma unroll
          for (int k = 0; k < H / 16; ++k) {
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) pk[i] = pack_bf16x2(f[16 * k + 2 * i] * inv, f[16 * k + 2 * i + 1] * inv);
            if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
              st_global_v8(dst + 16 * k, pk);
            } else {
              reinterpret_cast<uint4*>(dst)[2 * k] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
              reinterpret_cast<uint4*>(dst)[2 * k + 1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
          }
          if (t == 0) reinterpret_cast<float*>(ws_slot(ws, p, layer) + p.lse_off)[orow] = (m_row + log2f(L_row)) * 0.6931471805599453f;
        }
        // A CTA must not exit while a bulk copy still reads its staging tile: every rank has waited for the copies
        // addressed to it, so once all of them are here every copy is complete.
        cluster_arrive_relaxed();
        cluster_wait();
      }
    }
  }

  if (lane == 0) {
    stamp_end(p);
    if (abort_flag[0]) atomicExch(reinterpret_cast<int*>(ws), -4 /* KVC_ETIMEOUT */);   // (a warp's own waits are over)
  }
}

// ------------------------------------------------------------------------------------------------
// a2 score: one CTA per 128 candidate keys of one kv-head.  S^T = K_tile Q_obs^T puts keys on the
// TMEM lanes, so each thread owns one key and sums 2^(s*scale_log2 - lse2) over the observer
// columns in its own registers.  Observer rows are processed in groups of up to 256 columns.
// grid (ceil(n_cand/128), Hkv, nl), block 128, dynamic smem (D/64)*16 KB + (D/64)*32 KB + 1 KB.
struct TcSmemScore {
  uint64_t bar_k, bar_q, bar_s;
  uint32_t tmem_base;
  int wait_ctl[2];           // [0] abort flag, [1] wait limit in units of 1024 cycles (see mbar_wait)
  alignas(16) float lse2[256];
};

template <int D>
__global__ void __launch_bounds__(128) score_tc_kernel(const __grid_constant__ CUtensorMap tm_k,
                                                       const __grid_constant__ CUtensorMap tm_qobs,
                                                       char* __restrict__ ws, Geom p, int tok_per_group) {
  constexpr int NSUB = D / 64;
  constexpr uint32_t TMEM_COLS = 256;
  constexpr int kQSubBytes = 256 * 128;        // up to 256 observer rows x 128 B
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = smem;
  uint8_t* sQ = sK + NSUB * kSubTileBytes;
  __shared__ TcSmemScore sh;

  const int layer = blockIdx.z, g = blockIdx.y, key0 = blockIdx.x * 128;
  const int warp = threadIdx.x >> 5;
  char* slot = ws_slot(ws, p, layer);
  const float* lse = reinterpret_cast<const float*>(slot + p.lse_off);
  float* score = reinterpret_cast<float*>(slot + p.score_off) + static_cast<long long>(g) * p.cap;

  if (threadIdx.x == 0) {
    stamp_begin(p);
    mbar_init(&sh.bar_k, 1); mbar_init(&sh.bar_q, 1); mbar_init(&sh.bar_s, 1);
    sh.wait_ctl[0] = 0; sh.wait_ctl[1] = p.wait_limit_k;
    mbar_fence_init();
  }
  // observer rows beyond the last group's real rows are padding: keep them finite
  for (int i = threadIdx.x; i < NSUB * kQSubBytes / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(sQ)[i] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  if (warp == 0) {
    tmem_alloc(&sh.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sh.tmem_base;
  volatile int* abort_flag = sh.wait_ctl;
  const uint32_t lane_addr = static_cast<uint32_t>(warp * 32) << 16;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_qobs);
    mbar_expect_tx(&sh.bar_k, NSUB * kSubTileBytes);
    for (int sub = 0; sub < NSUB; ++sub)
      tma_load_4d(sK + sub * kSubTileBytes, &tm_k, &sh.bar_k, sub * 64, key0, g, layer);
  }
  // two sums, over the even and the odd 16-column pieces, as in the fused kernel: a launch of up to 256 observer rows may
  // take either form, and its scores must not depend on which
  float acc[2] = {0.f, 0.f};
  bool ok = true;
  const int n_groups = (p.w + tok_per_group - 1) / tok_per_group;
  int grp = 0, issued = 0;                                             // (thread 0: groups whose products have been issued)
  for (; grp < n_groups; ++grp) {
    const int t_first = p.n - p.w + grp * tok_per_group;               // first observer token of the group
    const int t_cnt = min(tok_per_group, p.n - t_first);
    const int cols = t_cnt * p.G;                                      // real observer columns
    const int n_mma = (cols + 15) & ~15;                               // MMA N: multiple of 16, <= 256
    // everyone is past the previous group's TMEM reads and smem reads, and all go on or, if a wait ran out, none
    tc_fence_before_sync();
    if (!__syncthreads_and(ok)) { ok = false; break; }
    for (int c = threadIdx.x; c < 256; c += blockDim.x) {
      float lv = INFINITY;                                             // padding column: 2^-inf = 0
      if (c < cols) lv = lse[static_cast<long long>(t_first + c / p.G) * p.Hq + g * p.G + c % p.G] * 1.4426950408889634f;
      sh.lse2[c] = lv;
    }
    if (threadIdx.x == 0) {
      // the box always spans tok_per_group tokens; tokens past n are zero-filled by TMA
      mbar_expect_tx(&sh.bar_q, NSUB * tok_per_group * p.G * 128);
      for (int sub = 0; sub < NSUB; ++sub)
        tma_load_4d(sQ + sub * kQSubBytes, &tm_qobs, &sh.bar_q, sub * 64, g * p.G, t_first, layer);
      if (grp == 0) ok = mbar_wait(&sh.bar_k, 0, abort_flag);
      ok = ok && mbar_wait(&sh.bar_q, grp & 1, abort_flag);
      if (ok) {
        tc_fence_after_sync();
        const uint32_t idesc = idesc_bf16_f32(128, n_mma, 0, 0);
        const uint32_t aK = smem_u32(sK), aQ = smem_u32(sQ);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
          mma_ss(tmem, smem_desc_sw128(aK + (kk / 4) * kSubTileBytes + (kk % 4) * 32, 16, 1024),
                 smem_desc_sw128(aQ + (kk / 4) * kQSubBytes + (kk % 4) * 32, 16, 1024), idesc, kk > 0);
        mma_commit(&sh.bar_s);
        ++issued;
      }
    }
    __syncwarp();
    __syncthreads();                                                   // lse2 visible
    ok = __all_sync(0xffffffffu, mbar_wait(&sh.bar_s, grp & 1, abort_flag));   // (a warp reads TMEM as one)
    if (!ok) continue;
    tc_fence_after_sync();
    for (int c0 = 0; c0 < n_mma; c0 += 32) {                           // the second half may be absent
      uint32_t sr[32];
      const bool two = c0 + 16 < n_mma;
      tmem_ld16(tmem + lane_addr + c0, sr);
      if (two) tmem_ld16(tmem + lane_addr + c0 + 16, sr + 16);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[0] += fast_exp2(fmaf(__uint_as_float(sr[i]), p.scale_log2, -sh.lse2[c0 + i]));
      if (two) {
#pragma unroll
        for (int i = 16; i < 32; ++i) acc[1] += fast_exp2(fmaf(__uint_as_float(sr[i]), p.scale_log2, -sh.lse2[c0 + i]));
      }
    }
  }
  const int key = key0 + threadIdx.x;
  if (ok && key < p.n_cand) score[key] = acc[0] + acc[1];
  // Thread 0 has given up: not before its loads and MMAs are complete does the block give up what they use.  (Asked without need
  // they cost 0.4 - 0.9 of the 36 - 41 us of a call with 384 or 448 observer rows.)
  if (threadIdx.x == 0 && __builtin_expect(!ok, 0)) {
    mbar_drain(&sh.bar_k, 0);
    mbar_drain(&sh.bar_q, (grp - 1) & 1);                              // (groups 0 .. grp - 1 have been loaded)
    if (issued > 0) mbar_drain(&sh.bar_s, (issued - 1) & 1);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0) stamp_end(p);
  if (threadIdx.x == 0 && sh.wait_ctl[0]) atomicExch(reinterpret_cast<int*>(ws), -4 /* KVC_ETIMEOUT */);
}

}  // namespace kvc
