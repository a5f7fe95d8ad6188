// CUDA-core kernels: fp32-accurate append + attention (a0, a1) and score (a2) for fp32 inputs
// (and, as a diagnostic, bf16 inputs).
#pragma once
#include "geom.cuh"
#include "ptx.cuh"

namespace kvc {

// Both kernels below are register-tiled products on the FMA pipes (packed fp32: one instruction, two IEEE fused
// multiply-adds).  A warp is a 4 x 8 grid of lanes: lane (rg, kg) holds rows rg, rg + 4, ... of the row tile and keys
// kg, kg + 8, ... of the key tile, so that an operand row is one 16-byte shared-memory read for four or eight lanes at
// once (row stride D + 4 floats: the distinct rows of one read lie on different banks) and feeds 2 .. 8 products.
static constexpr int kCcThreads = 256, kCcWarps = 8;

__device__ __forceinline__ ulonglong2 lds_f32x4(const float* s) { return *reinterpret_cast<const ulonglong2*>(s); }

// Eight or four consecutive elements to shared memory as fp32: fp32 asynchronously (cp.async), bf16 through registers.
// Both read through L2 only: the score kernel stages inputs in front of its dependency wait, where L1 may be stale.
template <typename T>
__device__ __forceinline__ void stage16(float* dst, const T* src) {
  if constexpr (sizeof(T) == 4) {
    cp_async16(dst, src);
  } else {
    const uint4 raw = __ldcg(reinterpret_cast<const uint4*>(src));
    reinterpret_cast<float4*>(dst)[0] = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                                                    __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
    reinterpret_cast<float4*>(dst)[1] = make_float4(__uint_as_float(raw.z << 16), __uint_as_float(raw.z & 0xffff0000u),
                                                    __uint_as_float(raw.w << 16), __uint_as_float(raw.w & 0xffff0000u));
  }
}

template <typename T> __device__ __forceinline__ void store4(T* dst, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* dst, float4 v) { *reinterpret_cast<float4*>(dst) = v; }
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* dst, float4 v) {
  *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
}

// ------------------------------------------------------------------------------------------------
// a0 + a1 on CUDA cores: append (Alg. 1: C <- C u (K_i, V_i)) and attention (Eq. 1), fp32 arithmetic throughout.
// The G query heads of a kv-head are stacked with the tokens (row = token * G + head), a CTA takes BM rows.  Its eight
// warps share the rows and split the KEYS: warp w of cluster rank s takes key tiles s*8 + w, + 8*S, ... with a running
// maximum, row sums and an output of its own, which are merged in shared memory at the end.  So no warp waits for
// another inside the loop, and a launch with few rows still fills the SMs.  Bound: with many rows the FMA pipe (4608
// rows, 1088 keys, d = 128: 48 us, 1.9 GFLOP at 39 TFLOP/s, where one key per lane and shuffled probabilities took
// 154 us), with few the latency of a step (256 rows, 192 keys, d = 64: 5.6 us against 23 us for 16 CTAs that each walked
// all keys), by device stamps.  The next K tile is fetched (cp.async) while the current one's
// P V is computed, the next V tile behind the scores.  Keys are the cache rows [0, n_c) followed by the block's own
// tokens, read from the inputs; the CTAs of a kv-head copy the block's rows into the cache on the side.
// grid (ceil(n*G/BM) * S, Hkv, nl), cluster (S,1,1) with S a power of two, block 256, dynamic smem AttnCc::kBytes.
template <int D, int BM>
struct AttnCc {
  static constexpr int KT = D == 128 ? 16 : 32;            // keys per warp and step
  static constexpr int KS = D + 4, PS = KT + 4;            // row strides (floats) of Q / K and of P
  static constexpr int kWarpFloats = KT * KS + KT * D;     // a warp's K and V tile; holds its O at the end
  static_assert(kWarpFloats >= BM * D, "a warp's O overlays its K and V tiles");
  static constexpr int kBytes = (BM * KS + kCcWarps * BM * PS + kCcWarps * kWarpFloats + 3 * kCcWarps * BM) * 4;
};

template <typename T, int D, int BM>
__global__ void __launch_bounds__(kCcThreads, 1) attn_cc_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                                const T* __restrict__ v, char* __restrict__ cache,
                                                                T* __restrict__ out, char* __restrict__ ws, Geom p, int S) {
  using L = AttnCc<D, BM>;
  constexpr int KT = L::KT, KS = L::KS, PS = L::PS, RT = BM / 4, JT = KT / 8, CT = D / 32;
  constexpr int EPC = 16 / (int)sizeof(T), CPR = D / EPC;  // elements per 16-byte piece, pieces per row
  constexpr int kUnrollS = D == 128 ? 8 : 4, kUnrollV = D == 128 ? 4 : 2;
  // (d = 128: 3 % faster than 4 and 2, although 32 rows per CTA then take all 255 registers and spill 8 bytes, bf16 inputs
  // 44; d = 64: slower)
  extern __shared__ __align__(16) float smem_f[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = lane >> 3, kg = lane & 7;
  float* sQ = smem_f;                                       // [BM][KS]; at the end this CTA's merged rows
  float* sP = sQ + BM * KS + warp * BM * PS;                // [BM][PS] of this warp
  float* bufs = sQ + BM * KS + kCcWarps * BM * PS;
  float* sK = bufs + warp * L::kWarpFloats;                 // [KT][KS]
  float* sV = sK + KT * KS;                                 // [KT][D]
  float* sM = bufs + kCcWarps * L::kWarpFloats;             // [8][BM] the warps' maxima, later their weights
  float* sL = sM + kCcWarps * BM;                           // [8][BM] row sums
  float* sA = sL + kCcWarps * BM;                           // [2][BM] merged maximum and sum

  const int layer = blockIdx.z, g = blockIdx.y;
  const int split = S > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tile = static_cast<int>(gridDim.x) / S - 1 - static_cast<int>(blockIdx.x) / S;   // longest rows first
  const int row0 = tile * BM, rows = p.n * p.G;
  char* blob = cache + layer * p.cache_ls;
  T* Kc = reinterpret_cast<T*>(blob) + static_cast<long long>(g) * p.cap * D;
  T* Vc = reinterpret_cast<T*>(blob + p.v_off) + static_cast<long long>(g) * p.cap * D;
  const long long in_stride = static_cast<long long>(p.Hkv) * D;
  const T* Kn = k + layer * p.kv_ls + static_cast<long long>(g) * D;
  const T* Vn = v + layer * p.kv_ls + static_cast<long long>(g) * D;
  const T* qb = q + layer * p.q_ls + static_cast<long long>(g) * p.G * D;
  auto row_off = [&](int r) { return (static_cast<long long>(r / p.G) * p.Hq + r % p.G) * D; };   // row r of q / out

  pdl_wait();                                               // the previous block's compaction is done with the cache
  // (after the wait: the score kernel reads the inputs and the old cache rows before its own)
  pdl_launch_dependents();
  if (threadIdx.x == 0) stamp_begin(p);

  const int kv_end = p.n_c + (min(row0 + BM, rows) - 1) / p.G + 1;     // keys the last row of this CTA sees
  const int n_tiles = (kv_end + KT - 1) / KT;
  // (rows past the last visible key: a copy of it, masked below)
  auto fetch = [&](float* dst, int stride, const T* cached, const T* fresh, int kt) {
    if (kt < n_tiles) {
#pragma unroll
      for (int i = 0; i < KT * CPR / 32; ++i) {
        const int r = (lane + 32 * i) / CPR, c = (lane + 32 * i) % CPR * EPC;
        const int key = min(kt * KT + r, kv_end - 1);
        const T* src = key < p.n_c ? cached + static_cast<long long>(key) * D : fresh + (key - p.n_c) * in_stride;
        stage16<T>(dst + r * stride + c, src + c);
      }
    }
    cp_async_commit();
  };
  const int step = S * kCcWarps;
  int kt = split * kCcWarps + warp;
  for (int i = threadIdx.x; i < BM * CPR; i += kCcThreads) {
    const int r = i / CPR, c = i % CPR * EPC;
    stage16<T>(sQ + r * KS + c, qb + row_off(min(row0 + r, rows - 1)) + c);
  }
  fetch(sK, KS, Kc, Kn, kt);
  fetch(sV, D, Vc, Vn, kt);
  // a0: warp w of CTA x copies tokens 8x + w, ...: one row of K and one of V each
  for (int t = blockIdx.x * kCcWarps + warp; t < p.n; t += gridDim.x * kCcWarps) {
    const long long dst = p.n_c + t;
    if (lane < CPR) {
      reinterpret_cast<uint4*>(Kc + dst * D)[lane] = reinterpret_cast<const uint4*>(Kn + t * in_stride)[lane];
      reinterpret_cast<uint4*>(Vc + dst * D)[lane] = reinterpret_cast<const uint4*>(Vn + t * in_stride)[lane];
    }
    if (lane == 0) reinterpret_cast<int*>(blob + p.pos_off)[static_cast<long long>(g) * p.cap + dst] = static_cast<int>(p.pos0 + t);
  }

  int lim[RT];                                              // visible keys of the thread's rows (causal inside the block)
  float m[RT], l[RT];
  uint64_t acc[RT][2 * CT];                                 // columns (kg + 8c)*4 .. +3 of every row, in pairs
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int r = row0 + rg + 4 * i;
    lim[i] = r < rows ? p.n_c + r / p.G + 1 : 0;
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 2 * CT; ++c) acc[i][c] = 0ull;
  }
  const int lim_min = row0 + BM <= rows ? p.n_c + row0 / p.G + 1 : 0;
  cp_async_wait<1>();                                       // Q and the first K tile have landed
  __syncthreads();

  for (; kt < n_tiles; kt += step) {
    cp_async_wait<1>();
    __syncwarp();
    uint64_t s2[RT][JT];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < JT; ++j) s2[i][j] = 0ull;
#pragma unroll kUnrollS
    for (int c = 0; c < D; c += 4) {
      ulonglong2 b[JT];
#pragma unroll
      for (int j = 0; j < JT; ++j) b[j] = lds_f32x4(sK + (kg + 8 * j) * KS + c);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const ulonglong2 a = lds_f32x4(sQ + (rg + 4 * i) * KS + c);
#pragma unroll
        for (int j = 0; j < JT; ++j) { s2[i][j] = fma_f32x2(a.x, b[j].x, s2[i][j]); s2[i][j] = fma_f32x2(a.y, b[j].y, s2[i][j]); }
      }
    }
    __syncwarp();
    fetch(sK, KS, Kc, Kn, kt + step);
    const bool masked = (kt + 1) * KT > lim_min;
    bool grew = false;
    float corr[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      float s[JT], mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < JT; ++j) {
        float lo, hi;
        f32x2_split(s2[i][j], lo, hi);
        s[j] = (lo + hi) * p.scale_log2;
        if (masked && kt * KT + kg + 8 * j >= lim[i]) s[j] = -INFINITY;
        mx = fmaxf(mx, s[j]);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(m[i], mx);
      const float m_use = m_new == -INFINITY ? 0.f : m_new;
      corr[i] = exp2f(m[i] - m_use);
      grew |= m_new > m[i];
      m[i] = m_new;
      l[i] *= corr[i];
#pragma unroll
      for (int j = 0; j < JT; ++j) {
        const float e = exp2f(s[j] - m_use);
        l[i] += e;
        sP[(rg + 4 * i) * PS + kg + 8 * j] = e;
      }
    }
    if (__any_sync(0xffffffffu, grew)) {
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const uint64_t f = f32x2(corr[i], corr[i]);
#pragma unroll
        for (int c = 0; c < 2 * CT; ++c) acc[i][c] = mul_f32x2(acc[i][c], f);
      }
    }
    cp_async_wait<1>();                                     // the V tile
    __syncwarp();
#pragma unroll kUnrollV
    for (int j = 0; j < KT; j += 4) {
      float4 pr[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) pr[i] = *reinterpret_cast<const float4*>(sP + (rg + 4 * i) * PS + j);
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        ulonglong2 vv[CT];
#pragma unroll
        for (int c = 0; c < CT; ++c) vv[c] = lds_f32x4(sV + (j + jj) * D + (kg + 8 * c) * 4);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float pv = jj == 0 ? pr[i].x : jj == 1 ? pr[i].y : jj == 2 ? pr[i].z : pr[i].w;
          const uint64_t pp = f32x2(pv, pv);
#pragma unroll
          for (int c = 0; c < CT; ++c) { acc[i][2 * c] = fma_f32x2(pp, vv[c].x, acc[i][2 * c]); acc[i][2 * c + 1] = fma_f32x2(pp, vv[c].y, acc[i][2 * c + 1]); }
        }
      }
    }
    __syncwarp();
    fetch(sV, D, Vc, Vn, kt + step);
  }
  cp_async_wait<0>();
  __syncwarp();

  // merge the warps' partial results: every warp leaves its O over its tiles, and (m, l) beside it
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int r = rg + 4 * i;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);
    if (kg == 0) { sM[warp * BM + r] = m[i]; sL[warp * BM + r] = l[i]; }
#pragma unroll
    for (int c = 0; c < CT; ++c) *reinterpret_cast<ulonglong2*>(sK + r * D + (kg + 8 * c) * 4) = make_ulonglong2(acc[i][2 * c], acc[i][2 * c + 1]);
  }
  __syncthreads();
  if (threadIdx.x < BM) {
    const int r = threadIdx.x;
    float mw[kCcWarps], ma = -INFINITY, sum = 0.f;
#pragma unroll
    for (int w = 0; w < kCcWarps; ++w) { mw[w] = sM[w * BM + r]; ma = fmaxf(ma, mw[w]); }
#pragma unroll
    for (int w = 0; w < kCcWarps; ++w) {
      const float wt = mw[w] == -INFINITY ? 0.f : exp2f(mw[w] - ma);   // -inf: the warp saw no key of the row
      sum = fmaf(wt, sL[w * BM + r], sum);
      sM[w * BM + r] = wt;
    }
    sA[r] = ma; sA[BM + r] = sum;
  }
  __syncthreads();
  T* ob = out + layer * p.out_ls + static_cast<long long>(g) * p.G * D;
  float* lse = reinterpret_cast<float*>(ws_slot(ws, p, layer) + p.lse_off) + g * p.G;
  auto write = [&](int r, int c, float4 o, float mx, float sum) {
    if (row0 + r >= rows) return;
    const float inv = 1.f / sum;
    store4<T>(ob + row_off(row0 + r) + c * 4, make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv));
    if (c == 0) lse[static_cast<long long>((row0 + r) / p.G) * p.Hq + (row0 + r) % p.G] = (mx + log2f(sum)) * 0.6931471805599453f;
  };
#pragma unroll 1
  for (int i = threadIdx.x; i < BM * D / 4; i += kCcThreads) {
    const int r = i / (D / 4), c = i % (D / 4);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kCcWarps; ++w) {
      const float wt = sM[w * BM + r];
      const float4 x = *reinterpret_cast<const float4*>(bufs + w * L::kWarpFloats + r * D + c * 4);
      o.x = fmaf(wt, x.x, o.x); o.y = fmaf(wt, x.y, o.y); o.z = fmaf(wt, x.z, o.z); o.w = fmaf(wt, x.w, o.w);
    }
    if (S == 1) write(r, c, o, sA[r], sA[BM + r]);
    else *reinterpret_cast<float4*>(sQ + r * KS + c * 4) = o;
  }
  if (S > 1) {                                              // merge over the cluster: rank s takes rows s, s + S, ...
    cluster_arrive(); cluster_wait();
#pragma unroll 1
    for (int i = threadIdx.x; i < BM / S * (D / 4); i += kCcThreads) {
      const int r = i / (D / 4) * S + split, c = i % (D / 4);
      // (all remote reads are issued before the first result is used: one at a time they cost 10 us at S = 8)
      float ma = -INFINITY, sum = 0.f, ms[8], ls[8];
      float4 xs[8];
#pragma unroll
      for (int s2 = 0; s2 < 8; ++s2) {
        const int src = s2 < S ? s2 : split;                // (S <= 8; the others repeat this rank's with weight zero)
        ms[s2] = dsmem_ld_f32(dsmem_addr(smem_u32(sA + r), src));
        ls[s2] = dsmem_ld_f32(dsmem_addr(smem_u32(sA + BM + r), src));
        xs[s2] = dsmem_ld_v4(dsmem_addr(smem_u32(sQ + r * KS + c * 4), src));
      }
#pragma unroll
      for (int s2 = 0; s2 < 8; ++s2) ma = fmaxf(ma, ms[s2]);
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s2 = 0; s2 < 8; ++s2) {
        const float wt = s2 >= S || ms[s2] == -INFINITY ? 0.f : exp2f(ms[s2] - ma);
        sum = fmaf(wt, ls[s2], sum);
        o.x = fmaf(wt, xs[s2].x, o.x); o.y = fmaf(wt, xs[s2].y, o.y); o.z = fmaf(wt, xs[s2].z, o.z); o.w = fmaf(wt, xs[s2].w, o.w);
      }
      write(r, c, o, ma, sum);
    }
    cluster_arrive(); cluster_wait();                       // nobody leaves while its rows are being read
  }
  __syncthreads();
  if (threadIdx.x == 0) stamp_end(p);
}

// ------------------------------------------------------------------------------------------------
// a2 score on CUDA cores (Eq. 4): score_j = sum over the w observer rows and the G heads of the
// group of 2^(s_ij*scale_log2 - lse2_i).  A CTA owns NK candidate keys; its eight warps take 16 observer rows each,
// 128 at a time, and their sums are added in a fixed order at the end.  Bound: loading the observer rows, then the
// FMA pipe (2 kv-heads x 1056 keys x 128 rows, d = 128: 7.9 us; one key per 16 threads took 65 us), of which all but the
// exponentials overlaps the attention's end (1 x 160 keys, d = 64: 3.2 -> 1.1 us behind the dependency wait).
// grid (ceil(n_cand/NK), Hkv, nl), block 256, dynamic smem score_cc_bytes.
static constexpr int kScoreCcRows = 128;
template <int D, int NK> constexpr int score_cc_bytes() { return ((NK + kScoreCcRows) * (D + 4) + kScoreCcRows + kCcWarps * NK) * 4; }

template <typename T, int D, int NK>
__global__ void __launch_bounds__(kCcThreads) score_cc_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                              const char* __restrict__ cache,
                                                              char* __restrict__ ws, Geom p) {
  constexpr int KS = D + 4, RT = 4, JT = NK / 8;
  constexpr int EPC = 16 / (int)sizeof(T), CPR = D / EPC;
  extern __shared__ __align__(16) float smem_f[];
  float* sK = smem_f;                          // [NK][KS]
  float* sQ = sK + NK * KS;                    // [128][KS]
  float* sL = sQ + kScoreCcRows * KS;          // [128]
  float* sS = sL + kScoreCcRows;               // [8][NK] the warps' sums
  const int layer = blockIdx.z, g = blockIdx.y, key0 = blockIdx.x * NK;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = lane >> 3, kg = lane & 7;
  const char* blob = cache + layer * p.cache_ls;
  const T* Kc = reinterpret_cast<const T*>(blob) + static_cast<long long>(g) * p.cap * D;
  const T* qb = q + layer * p.q_ls;
  char* slot = ws_slot(ws, p, layer);
  const float* lse = reinterpret_cast<const float*>(slot + p.lse_off);
  float* score = reinterpret_cast<float*>(slot + p.score_off) + static_cast<long long>(g) * p.cap;

  // Keys, observer rows and the first group's products come before the dependency wait: the inputs and the cache rows
  // below n_c are complete (the attention kernel allows this launch after its own wait), the block's keys are read from
  // the input.  Only the exponentials need what the attention kernel leaves.
  pdl_launch_dependents();
  if (threadIdx.x == 0 && p.stamp_early) stamp_begin(p);
  const long long in_stride = static_cast<long long>(p.Hkv) * D;
  const T* Kn = k + layer * p.kv_ls + static_cast<long long>(g) * D;
  for (int i = threadIdx.x; i < NK * CPR; i += kCcThreads) {
    const int r = i / CPR, c = i % CPR * EPC, key = min(key0 + r, p.n_cand - 1);
    stage16<T>(sK + r * KS + c, (key < p.n_sc ? Kc + static_cast<long long>(key) * D : Kn + (key - p.n_sc) * in_stride) + c);
  }
  const int rows = p.w * p.G;
  float acc[JT];
#pragma unroll
  for (int j = 0; j < JT; ++j) acc[j] = 0.f;
  for (int r0 = 0; r0 < rows; r0 += kScoreCcRows) {
    const int cnt = min(kScoreCcRows, rows - r0);
    if (r0) __syncthreads();
    auto token_head = [&](int r) { return static_cast<long long>(p.n - p.w + r / p.G) * p.Hq + g * p.G + r % p.G; };
    for (int i = threadIdx.x; i < cnt * CPR; i += kCcThreads) {
      const int r = i / CPR, c = i % CPR * EPC;
      stage16<T>(sQ + r * KS + c, qb + token_head(r0 + r) * D + c);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const int w0 = warp * 16;                  // this warp's rows of the group (rows past the last: a copy of it, not summed)
    uint64_t s2[RT][JT];
    if (w0 < cnt) {
      const float* qr[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        qr[i] = sQ + min(w0 + rg + 4 * i, cnt - 1) * KS;
#pragma unroll
        for (int j = 0; j < JT; ++j) s2[i][j] = 0ull;
      }
#pragma unroll 4
      for (int c = 0; c < D; c += 4) {
        ulonglong2 b[JT];
#pragma unroll
        for (int j = 0; j < JT; ++j) b[j] = lds_f32x4(sK + (kg + 8 * j) * KS + c);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const ulonglong2 a = lds_f32x4(qr[i] + c);
#pragma unroll
          for (int j = 0; j < JT; ++j) { s2[i][j] = fma_f32x2(a.x, b[j].x, s2[i][j]); s2[i][j] = fma_f32x2(a.y, b[j].y, s2[i][j]); }
        }
      }
    }
    if (r0 == 0) {
      pdl_wait();
      if (threadIdx.x == 0) stamp_begin(p);
    }
    if (threadIdx.x < cnt) sL[threadIdx.x] = lse[token_head(r0 + threadIdx.x)] * 1.4426950408889634f;
    __syncthreads();
    if (w0 < cnt) {
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = w0 + rg + 4 * i;
        if (r < cnt) {
#pragma unroll
          for (int j = 0; j < JT; ++j) {
            float lo, hi;
            f32x2_split(s2[i][j], lo, hi);
            acc[j] += exp2f((lo + hi) * p.scale_log2 - sL[r]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < JT; ++j) {
    acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], 8);
    acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], 16);
    if (rg == 0) sS[warp * NK + kg + 8 * j] = acc[j];
  }
  __syncthreads();
  if (threadIdx.x < NK && key0 + threadIdx.x < p.n_cand) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kCcWarps; ++w) t += sS[w * NK + threadIdx.x];
    score[key0 + threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) stamp_end(p);
}

// ------------------------------------------------------------------------------------------------
// Self-test of the bounded wait: one CTA waits on an mbarrier that nobody will ever arrive on.  With a wait limit
// of a few thousand cycles the wait gives up, the CTA passes its barrier, records KVC_ETIMEOUT in the status word
// exactly as the production kernels do, and returns.  Nothing in it can wait longer than the limit.
// grid 1, block 128.
__global__ void __launch_bounds__(128) wait_timeout_selftest_kernel(char* __restrict__ ws, int wait_limit_k) {
  __shared__ uint64_t bar;
  __shared__ int wait_ctl[2];
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    wait_ctl[0] = 0; wait_ctl[1] = wait_limit_k;
    mbar_fence_init();
  }
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0, wait_ctl);          // phase 0 never completes: returns false after the limit
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || wait_ctl[0])) atomicExch(reinterpret_cast<int*>(ws), -4 /* KVC_ETIMEOUT */);
}

}  // namespace kvc
