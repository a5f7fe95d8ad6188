// Host side of the kvc C ABI (see include/kvc.h): argument checks, launch geometry, TMA tensor
// maps, kernel launches on the caller's stream.  Allocates no device memory.
#include "../../include/kvc.h"

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "geom.cuh"
#include "kernels_cc.cuh"
#include "kernels_tc.cuh"
#include "compress.cuh"

using kvc::Geom;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct kvc_ctx {
  uint32_t magic;
  kvc_config cfg;
  int G, cap, w_cfg;
  float scale;
  size_t elem, blob_bytes, v_off, pos_off;
  size_t ws_slot_bytes, ws_bytes, lse_off, score_off, msrc_off, mdst_off, mcount_off;
  std::vector<int> len;          // current cache length per layer, -1 = never reset
  long long launches;
  EncodeTiledFn encode;
  bool use_tc;
  bool profiling;
  int wait_limit_k;              // limit of the kernels' waits, in units of 1024 clock cycles
  struct Prof { int kind; cudaEvent_t a, b; };
  std::vector<Prof> prof;
  // device-side time stamps (kvc_profile_device): the caller's record buffer, its capacity, the kind of every launch so far
  unsigned long long* stamps_dev;
  long long stamps_cap;
  std::vector<int> stamp_kind;
  // KVC_FLAG_ASYNC_COMPRESS: the side streams, per layer an event after its attention and one after its
  // compress kernel, and whether that compress may still be running (host objects, created on first use)
  static constexpr int kSideStreams = 2;     // layers alternate between them: consecutive compress kernels may overlap
  cudaStream_t side[kSideStreams];
  std::vector<cudaEvent_t> ev_attn, ev_comp;
  std::vector<char> pending;
  // kvc_prefill_chunk_host: the stream that carries the host-to-device copies, per staging half an event after its
  // copies (recorded there) and one after the block that read it (recorded on the caller's stream); call counter
  cudaStream_t copy_in, copy_out;
  cudaEvent_t ev_in[2], ev_free[2], ev_out[2];
  unsigned host_calls;
  char err[512];
};

static const uint32_t kMagic = 0x6b766331u;   // "kvc1"

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static int fail(kvc_ctx* c, int code, const char* fmt, ...) {
  if (c) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(c->err, sizeof(c->err), fmt, ap);
    va_end(ap);
  }
  return code;
}

static bool live(const kvc_ctx* c) { return c && c->magic == kMagic; }

extern "C" int kvc_create(const kvc_config* cfg, kvc_ctx** out) {
  if (!out) return KVC_EINVAL;
  *out = nullptr;
  if (!cfg) return KVC_EINVAL;
  if (cfg->n_layers < 1 || cfg->n_kv_heads < 1 || cfg->n_q_heads < 1) return KVC_EINVAL;
  if (cfg->n_q_heads % cfg->n_kv_heads != 0) return KVC_EINVAL;
  if (cfg->head_dim != 64 && cfg->head_dim != 128) return KVC_EINVAL;
  if (cfg->dtype != KVC_F32 && cfg->dtype != KVC_BF16) return KVC_EINVAL;
  if (cfg->budget < 1 || cfg->max_chunk < 1) return KVC_EINVAL;
  if (cfg->policy != KVC_SCORE_ATTN && cfg->policy != KVC_SCORE_KEYDIFF) return KVC_EINVAL;
  if (cfg->obs_window < 0) return KVC_EINVAL;
  if (!(cfg->softmax_scale >= 0.f) || isinf(cfg->softmax_scale)) return KVC_EINVAL;
  const int w = cfg->obs_window == 0 ? 32 : cfg->obs_window;
  if (w > cfg->budget) return KVC_EINVAL;                 // the protected window must fit the budget
  const int G = cfg->n_q_heads / cfg->n_kv_heads;
  if (G > 128) return KVC_EINVAL;
  if (cfg->device < 0 || cfg->device >= 64) return KVC_EINVAL;   // per-device tables below hold 64 ordinals
  if ((long long)cfg->budget + cfg->max_chunk > (1ll << 30)) return KVC_EINVAL;

  kvc_ctx* c = new (std::nothrow) kvc_ctx();
  if (!c) return KVC_EINVAL;
  c->magic = kMagic;
  c->cfg = *cfg;
  c->G = G;
  c->w_cfg = w;
  c->scale = cfg->softmax_scale > 0.f ? cfg->softmax_scale : 1.0f / sqrtf((float)cfg->head_dim);
  c->cap = (int)align_up((size_t)cfg->budget + cfg->max_chunk, 128);
  c->elem = cfg->dtype == KVC_F32 ? 4 : 2;
  const size_t kv_bytes = (size_t)cfg->n_kv_heads * c->cap * cfg->head_dim * c->elem;
  c->v_off = kv_bytes;
  c->pos_off = 2 * kv_bytes;
  c->blob_bytes = align_up(2 * kv_bytes + (size_t)cfg->n_kv_heads * c->cap * 4, 1024);
  size_t o = 0;
  // (lse has room for a first block of up to B tokens: the hybrid schedule of Sec. 5 (Budgeting) fills an empty cache in one pass)
  const size_t lse_rows = cfg->max_chunk > cfg->budget ? cfg->max_chunk : cfg->budget;
  c->lse_off = o;    o = align_up(o + lse_rows * cfg->n_q_heads * 4, 256);
  c->score_off = o;  o = align_up(o + (size_t)cfg->n_kv_heads * c->cap * 4, 256);
  c->msrc_off = o;   o = align_up(o + (size_t)cfg->n_kv_heads * cfg->max_chunk * 4, 256);
  c->mdst_off = o;   o = align_up(o + (size_t)cfg->n_kv_heads * cfg->max_chunk * 4, 256);
  c->mcount_off = o; o = align_up(o + (size_t)cfg->n_kv_heads * 4, 256);
  c->ws_slot_bytes = o;
  c->ws_bytes = kvc::kWsHeaderBytes + o * cfg->n_layers;
  c->len.assign(cfg->n_layers, -1);
  c->launches = 0;
  c->encode = nullptr;
  c->use_tc = cfg->dtype == KVC_BF16 && !(cfg->flags & KVC_FLAG_CUDA_CORES);
  c->profiling = false;
  c->stamps_dev = nullptr;
  c->stamps_cap = 0;
  c->wait_limit_k = kvc::kDefaultWaitLimitK;
  for (auto& s : c->side) s = nullptr;
  c->pending.assign(cfg->n_layers, 0);
  c->copy_in = c->copy_out = nullptr;
  for (int i = 0; i < 2; ++i) { c->ev_in[i] = nullptr; c->ev_free[i] = nullptr; c->ev_out[i] = nullptr; }
  c->host_calls = 0;
  c->err[0] = 0;
  *out = c;
  return KVC_OK;
}

static void drop_events(kvc_ctx* c) {
  for (auto& p : c->prof) { cudaEventDestroy(p.a); cudaEventDestroy(p.b); }
  c->prof.clear();
}

extern "C" int kvc_profile_enable(kvc_ctx* c, int on) {
  if (!live(c)) return KVC_ESTATE;
  c->profiling = on != 0;
  if (!on) drop_events(c);
  return KVC_OK;
}

extern "C" int kvc_profile_read(kvc_ctx* c, double* ms, long long* launches) {
  if (!live(c)) return KVC_ESTATE;
  if (!ms || !launches) return KVC_EINVAL;
  int rc = KVC_OK;
  for (auto& p : c->prof) {
    float t = 0.f;
    cudaError_t e = cudaEventSynchronize(p.b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, p.a, p.b);
    if (e != cudaSuccess) { rc = fail(c, KVC_ECUDA, "profile event: %s", cudaGetErrorString(e)); break; }
    ms[p.kind] += t;
    launches[p.kind] += 1;
  }
  drop_events(c);
  return rc;
}

extern "C" int kvc_profile_device(kvc_ctx* c, void* records, long long capacity, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  c->stamp_kind.clear();
  c->stamps_dev = nullptr;
  c->stamps_cap = 0;
  if (!records) return KVC_OK;
  if (capacity < 1 || (reinterpret_cast<uintptr_t>(records) & 15)) return fail(c, KVC_EINVAL, "records misaligned or capacity < 1");
  // every record starts as {begin = all ones, end = 0}: the kernels keep the minimum and the maximum
  cudaError_t e = cudaMemsetAsync(records, 0, (size_t)capacity * 16, (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaMemset2DAsync(records, 16, 0xff, 8, (size_t)capacity, (cudaStream_t)stream);
  if (e != cudaSuccess) return fail(c, KVC_ECUDA, "cudaMemsetAsync(records): %s", cudaGetErrorString(e));
  c->stamps_dev = (unsigned long long*)records;
  c->stamps_cap = capacity;
  return KVC_OK;
}

extern "C" int kvc_profile_device_read(kvc_ctx* c, const void* records_host, double* ms, long long* launches, double* span_ms) {
  if (!live(c)) return KVC_ESTATE;
  if (!records_host || !ms || !launches) return KVC_EINVAL;
  const unsigned long long* r = (const unsigned long long*)records_host;
  unsigned long long first = ~0ull, last = 0;
  for (size_t i = 0; i < c->stamp_kind.size(); ++i) {
    const unsigned long long b = r[2 * i], e = r[2 * i + 1];
    if (b == ~0ull || e < b) continue;                    // a launch whose CTAs never stamped (nothing to do)
    ms[c->stamp_kind[i]] += (double)(e - b) * 1e-6;
    launches[c->stamp_kind[i]] += 1;
    if (b < first) first = b;
    if (e > last) last = e;
  }
  if (span_ms) *span_ms = last > first ? (double)(last - first) * 1e-6 : 0.0;
  c->stamp_kind.clear();
  return KVC_OK;
}

// The record of the next launch of the given kind (null when device stamps are off or the buffer is full).
static unsigned long long* next_stamp(kvc_ctx* c, int kind) {
  if (!c->stamps_dev || (long long)c->stamp_kind.size() >= c->stamps_cap) return nullptr;
  c->stamp_kind.push_back(kind);
  return c->stamps_dev + 2 * (c->stamp_kind.size() - 1);
}

// Brackets one kernel launch with events when profiling is on.
struct ProfScope {
  kvc_ctx* c; cudaStream_t st; cudaEvent_t a, b; bool on;
  ProfScope(kvc_ctx* c_, int kind, cudaStream_t st_) : c(c_), st(st_), a(nullptr), b(nullptr), on(c_->profiling) {
    if (!on) return;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) { on = false; return; }
    cudaEventRecord(a, st);
    c->prof.push_back({kind, a, b});
  }
  ~ProfScope() { if (on) cudaEventRecord(b, st); }
};

// Makes `st` wait for the compress kernels of layers [l0, l1) that still run on the side stream.
static int wait_pending(kvc_ctx* c, int l0, int l1, cudaStream_t st) {
  for (int l = l0; l < l1; ++l) {
    if (!c->pending[l]) continue;
    cudaError_t e = cudaStreamWaitEvent(st, c->ev_comp[l], 0);
    if (e != cudaSuccess) return fail(c, KVC_ECUDA, "cudaStreamWaitEvent: %s", cudaGetErrorString(e));
    c->pending[l] = 0;
  }
  return KVC_OK;
}

// Makes `st` wait for the compress kernels that still use workspace slots [s0, s1) (slot l: layer l's).  They stay pending: a
// later call or kvc_join, perhaps on another stream, waits for them too.  One left over from before a capture of `st` began
// cannot be waited for inside it: the host does.
static int wait_slots(kvc_ctx* c, int s0, int s1, cudaStream_t st) {
  for (int l = s0; l < s1; ++l) {
    if (!c->pending[l]) continue;
    cudaStreamCaptureStatus here = cudaStreamCaptureStatusNone, there = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &here);
    if (e == cudaSuccess) e = cudaStreamIsCapturing(c->side[l % kvc_ctx::kSideStreams], &there);
    if (e == cudaSuccess && here != cudaStreamCaptureStatusNone && there == cudaStreamCaptureStatusNone) {
      cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
      (void)cudaThreadExchangeStreamCaptureMode(&mode);
      e = cudaEventSynchronize(c->ev_comp[l]);
      (void)cudaThreadExchangeStreamCaptureMode(&mode);
      if (e == cudaSuccess) c->pending[l] = 0;
    } else if (e == cudaSuccess) {
      e = cudaStreamWaitEvent(st, c->ev_comp[l], 0);
    }
    if (e != cudaSuccess) return fail(c, KVC_ECUDA, "wait for workspace slot %d: %s", l, cudaGetErrorString(e));
  }
  return KVC_OK;
}

static int ensure_side_stream(kvc_ctx* c) {
  if (c->side[0]) return KVC_OK;                             // set last: marks a complete set of events and streams
  cudaError_t e = cudaSuccess;
  c->ev_attn.resize(c->cfg.n_layers, nullptr);
  c->ev_comp.resize(c->cfg.n_layers, nullptr);
  for (int l = 0; l < c->cfg.n_layers; ++l) {
    if (!c->ev_attn[l] && (e = cudaEventCreateWithFlags(&c->ev_attn[l], cudaEventDisableTiming)) != cudaSuccess) c->ev_attn[l] = nullptr;
    if (e == cudaSuccess && !c->ev_comp[l] && (e = cudaEventCreateWithFlags(&c->ev_comp[l], cudaEventDisableTiming)) != cudaSuccess) c->ev_comp[l] = nullptr;
    if (e != cudaSuccess) return fail(c, KVC_ECUDA, "cudaEventCreate: %s", cudaGetErrorString(e));
  }
  for (int i = kvc_ctx::kSideStreams - 1; i >= 0; --i) {
    if (c->side[i]) continue;
    if ((e = cudaStreamCreateWithFlags(&c->side[i], cudaStreamNonBlocking)) != cudaSuccess) {
      c->side[i] = nullptr;
      return fail(c, KVC_ECUDA, "cudaStreamCreate: %s", cudaGetErrorString(e));
    }
  }
  return KVC_OK;
}

extern "C" int kvc_join(kvc_ctx* c, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  return wait_pending(c, 0, c->cfg.n_layers, (cudaStream_t)stream);
}

extern "C" int kvc_destroy(kvc_ctx* c) {
  if (!live(c)) return KVC_ESTATE;
  {
    for (auto s : c->side) if (s) cudaStreamSynchronize(s);
    for (auto ev : c->ev_attn) if (ev) cudaEventDestroy(ev);
    for (auto ev : c->ev_comp) if (ev) cudaEventDestroy(ev);
    c->ev_attn.clear(); c->ev_comp.clear();
    for (auto& s : c->side) { if (s) cudaStreamDestroy(s); s = nullptr; }
    if (c->copy_out) { cudaStreamSynchronize(c->copy_out); cudaStreamDestroy(c->copy_out); c->copy_out = nullptr; }
    if (c->copy_in) { cudaStreamSynchronize(c->copy_in); cudaStreamDestroy(c->copy_in); c->copy_in = nullptr; }
    for (int i = 0; i < 2; ++i) {
      if (c->ev_in[i]) cudaEventDestroy(c->ev_in[i]);
      if (c->ev_free[i]) cudaEventDestroy(c->ev_free[i]);
      if (c->ev_out[i]) cudaEventDestroy(c->ev_out[i]);
      c->ev_in[i] = c->ev_free[i] = c->ev_out[i] = nullptr;
    }
  }
  drop_events(c);
  c->magic = 0;
  delete c;
  return KVC_OK;
}

extern "C" const char* kvc_last_error(const kvc_ctx* c) { return live(c) ? c->err : "invalid context"; }
extern "C" long long kvc_launch_count(const kvc_ctx* c) { return live(c) ? c->launches : -1; }

extern "C" int kvc_cache_nbytes(const kvc_ctx* c, size_t* per_layer, size_t* workspace) {
  if (!live(c)) return KVC_ESTATE;
  if (per_layer) *per_layer = c->blob_bytes;
  if (workspace) *workspace = c->ws_bytes;
  return KVC_OK;
}

extern "C" int kvc_kv_bytes(const kvc_ctx* c, long long seq_len, size_t* logical, size_t* physical,
                            size_t* uncompressed) {
  if (!live(c)) return KVC_ESTATE;
  if (seq_len < 0) return KVC_EINVAL;
  // Eq. 2: 2 x layers x heads x dim_head x precision x sequence length
  const size_t per_tok = 2 * (size_t)c->cfg.n_layers * c->cfg.n_kv_heads * c->cfg.head_dim * c->elem;
  if (logical) *logical = per_tok * c->cfg.budget;
  if (physical) *physical = per_tok * c->cap;
  if (uncompressed) *uncompressed = per_tok * (size_t)seq_len;
  return KVC_OK;
}

static int check_cuda(kvc_ctx* c, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return KVC_OK;
  return fail(c, KVC_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

extern "C" int kvc_reset(kvc_ctx* c, int layer, int n_layers, void* cache, size_t cache_layer_stride, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (layer < 0 || n_layers < 1 || layer + n_layers > c->cfg.n_layers) return fail(c, KVC_EINVAL, "layer range");
  if (!cache || !aligned16(cache)) return fail(c, KVC_EINVAL, "cache pointer null or misaligned");
  if (n_layers > 1 && (cache_layer_stride < c->blob_bytes || cache_layer_stride % 16)) return fail(c, KVC_EINVAL, "cache_layer_stride");
  cudaStream_t st = (cudaStream_t)stream;
  if (int rc = wait_pending(c, layer, layer + n_layers, st)) return rc;
  // one fill for all layers: a fill per layer costs 2.7 us of host time and a gap on the GPU each
  const bool gaps = n_layers > 1 && cache_layer_stride != c->blob_bytes;
  const cudaError_t e = gaps ? cudaMemset2DAsync(cache, cache_layer_stride, 0, c->blob_bytes, n_layers, st)
                             : cudaMemsetAsync(cache, 0, c->blob_bytes * n_layers, st);
  if (int rc = check_cuda(c, e, "cudaMemsetAsync")) return rc;
  for (int i = 0; i < n_layers; ++i) c->len[layer + i] = 0;
  return KVC_OK;
}

extern "C" int kvc_workspace_init(kvc_ctx* c, void* workspace, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (!workspace || !aligned16(workspace)) return fail(c, KVC_EINVAL, "workspace pointer null or misaligned");
  return check_cuda(c, cudaMemsetAsync(workspace, 0, kvc::kWsHeaderBytes, (cudaStream_t)stream), "cudaMemsetAsync");
}

extern "C" int kvc_cache_view(const kvc_ctx* c, int layer, void* cache, kvc_view* v) {
  if (!live(c)) return KVC_ESTATE;
  if (!v || !cache || layer < 0 || layer >= c->cfg.n_layers) return KVC_EINVAL;
  if (c->len[layer] < 0) return KVC_ESTATE;
  v->k = cache;
  v->v = (char*)cache + c->v_off;
  v->pos = (int*)((char*)cache + c->pos_off);
  v->len = c->len[layer];
  v->cap = c->cap;
  v->n_kv_heads = c->cfg.n_kv_heads;
  v->head_dim = c->cfg.head_dim;
  v->dtype = c->cfg.dtype;
  return KVC_OK;
}

extern "C" int kvc_workspace_view(const kvc_ctx* c, void* workspace, int slot, float** lse, float** score) {
  if (!live(c)) return KVC_ESTATE;
  if (!workspace || slot < 0 || slot >= c->cfg.n_layers) return KVC_EINVAL;
  char* s = (char*)workspace + kvc::kWsHeaderBytes + (size_t)slot * c->ws_slot_bytes;
  if (lse) *lse = (float*)(s + c->lse_off);
  if (score) *score = (float*)(s + c->score_off);
  return KVC_OK;
}

extern "C" int kvc_move_counts(const kvc_ctx* c, void* workspace, int slot, int** counts) {
  if (!live(c)) return KVC_ESTATE;
  if (!workspace || !counts || slot < 0 || slot >= c->cfg.n_layers) return KVC_EINVAL;
  *counts = (int*)((char*)workspace + kvc::kWsHeaderBytes + (size_t)slot * c->ws_slot_bytes + c->mcount_off);
  return KVC_OK;
}

extern "C" int kvc_set_wait_limit(kvc_ctx* c, long long cycles) {
  if (!live(c)) return KVC_ESTATE;
  if (cycles < 1024 || cycles > (1ll << 40)) return fail(c, KVC_EINVAL, "wait limit %lld outside [1024, 2^40] cycles", cycles);
  c->wait_limit_k = (int)(cycles >> 10);
  return KVC_OK;
}

extern "C" int kvc_selftest_wait_timeout(kvc_ctx* c, void* workspace, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (!workspace || !aligned16(workspace)) return fail(c, KVC_EINVAL, "workspace pointer null or misaligned");
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != c->cfg.device)
    return fail(c, KVC_ESTATE, "current CUDA device %d is not the context's device %d", dev, c->cfg.device);
  // never more than about 2^21 cycles (a millisecond): the kernel exists to run into its limit
  const int limit_k = c->wait_limit_k < 2048 ? c->wait_limit_k : 2048;
  kvc::wait_timeout_selftest_kernel<<<1, 128, 0, (cudaStream_t)stream>>>((char*)workspace, limit_k);
  c->launches++;
  return check_cuda(c, cudaGetLastError(), "self-test launch");
}

extern "C" int kvc_status(kvc_ctx* c, void* workspace, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (!workspace) return KVC_EINVAL;
  int word = 0;
  int rc = wait_pending(c, 0, c->cfg.n_layers, (cudaStream_t)stream);
  if (rc) return rc;
  rc = check_cuda(c, cudaMemcpyAsync(&word, workspace, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream), "cudaMemcpyAsync");
  if (rc) return rc;
  rc = check_cuda(c, cudaStreamSynchronize((cudaStream_t)stream), "cudaStreamSynchronize");
  if (rc) return rc;
  if (word != 0) return fail(c, word == KVC_ETIMEOUT ? KVC_ETIMEOUT : KVC_ECUDA, "device status word %d", word);
  return KVC_OK;
}

// ------------------------------------------------------------------------------------------------
static int get_encoder(kvc_ctx* c) {
  if (c->encode) return KVC_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn)
    return fail(c, KVC_ECUDA, "cuTensorMapEncodeTiled entry point unavailable: %s", cudaGetErrorString(e));
  c->encode = (EncodeTiledFn)fn;
  return KVC_OK;
}

// bf16 4-D tensor map with 128-byte swizzle; dims/box innermost first, strides in bytes for dims 1..3.
static int make_map(kvc_ctx* c, CUtensorMap* m, const void* base, const uint64_t dims[4], const uint64_t strides[3],
                    const uint32_t box[4]) {
  cuuint64_t gd[4] = {dims[0], dims[1], dims[2], dims[3]};
  cuuint64_t gs[3] = {strides[0], strides[1], strides[2]};
  cuuint32_t bx[4] = {box[0], box[1], box[2], box[3]};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = c->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gd, gs, bx, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fail(c, KVC_ECUDA, "cuTensorMapEncodeTiled failed (%d): dims %llu %llu %llu %llu box %u %u %u %u", (int)r,
                (unsigned long long)dims[0], (unsigned long long)dims[1], (unsigned long long)dims[2],
                (unsigned long long)dims[3], box[0], box[1], box[2], box[3]);
  return KVC_OK;
}

// cudaFuncSetAttribute acts on the current device only: every kernel that opts into more dynamic shared memory keeps
// one flag per device ordinal (the caller has checked that the current device is the context's).
static const int kMaxDevices = 64;
template <typename Kernel>
static cudaError_t opt_in_smem(Kernel kernel, int bytes, bool* done_per_device, int dev) {
  if (done_per_device[dev]) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done_per_device[dev] = true;
  return e;
}

// Launch attributes shared by the PDL-aware kernels: an optional cluster size and, unless disabled,
// programmatic stream serialization (the kernel may start while its predecessor drains; it calls
// griddepcontrol.wait before it touches anything the predecessor wrote or still reads).
struct LaunchAttrs {
  cudaLaunchAttribute at[2];
  int n;
  LaunchAttrs(int cluster_x, bool pdl) : n(0) {
    if (cluster_x > 0) {
      at[n].id = cudaLaunchAttributeClusterDimension;
      at[n].val.clusterDim.x = cluster_x; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
      ++n;
    }
    if (pdl) {
      at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[n].val.programmaticStreamSerializationAllowed = 1;
      ++n;
    }
  }
};

template <typename T, int D, int BM>
static cudaError_t launch_cc_attn_bm(const Geom& g, int dev, const void* q, const void* k, const void* v, void* cache, void* out,
                                     void* ws, int S, bool pdl, cudaStream_t st) {
  using L = kvc::AttnCc<D, BM>;
  static bool attr_set[kMaxDevices] = {};
  if (cudaError_t e = opt_in_smem(kvc::attn_cc_kernel<T, D, BM>, L::kBytes, attr_set, dev)) return e;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3((int)(((long long)g.n * g.G + BM - 1) / BM) * S, g.Hkv, g.nl);
  lc.blockDim = dim3(kvc::kCcThreads, 1, 1);
  lc.dynamicSmemBytes = L::kBytes;
  lc.stream = st;
  LaunchAttrs la(S, pdl);
  lc.attrs = la.at;
  lc.numAttrs = la.n;
  return cudaLaunchKernelEx(&lc, kvc::attn_cc_kernel<T, D, BM>, (const T*)q, (const T*)k, (const T*)v, (char*)cache, (T*)out,
                            (char*)ws, g, S);
}
// Rows per CTA (BM) and key split (S) of the CUDA-core attention, by a model of its duration fitted to device stamps
// of all twelve shapes on nine configurations (128 .. 4608 rows, 192 .. 2080 keys): a step (a key tile per warp) costs
// 3.1 / 4.2 / 7 us at BM = 8 / 16 / 32, a CTA 3 us around its steps, the merge over a cluster 1.5 us more, and an SM
// holds one CTA (clusters of 4 and 8 find room for 32 and 14 of them at a time).  E.g. 128 rows, 2080 keys: BM 16, S 8
// 14.2 us against 41.1 (BM 8, S 1); 4608 rows, 1088 keys: BM 16, S 1 51.8 against 69.1 (BM 8) and 58.2 (BM 32);
// 3136 rows, 708 keys: BM 32, S 1 44.3 against 46.4 (BM 16).  The model's choice was the fastest shape or within 3 %.
template <typename T, int D>
static cudaError_t launch_cc_attn(const Geom& g, int dev, const void* q, const void* k, const void* v, void* cache, void* out,
                                  void* ws, bool allow_split, bool pdl, cudaStream_t st) {
  constexpr int KT = kvc::AttnCc<D, 8>::KT;
  const long long rows = (long long)g.n * g.G, heads = (long long)g.Hkv * g.nl;
  const int bms[3] = {32, 16, 8}, capacity[4] = {kvc::kNumSMs, kvc::kNumSMs, 128, 112};
  const double step_us[3] = {7.0, 4.2, 3.1};
  int BM = 32, S = 1;
  double best = 0.0;
  for (int b = 0; b < 3; ++b) {
    const long long base = (rows + bms[b] - 1) / bms[b] * heads;
    for (int s = 0; s < (allow_split ? 4 : 1); ++s) {
      if (s > 0 && (base << s) > capacity[s]) break;
      const long long waves = ((base << s) + capacity[s] - 1) / capacity[s];
      const int keys = waves > 1 ? g.n_c + g.n / 2 : g.n_c + g.n;      // the longest row, or the average over waves
      const int per_step = KT * (kvc::kCcWarps << s);
      const double est = (double)waves * ((keys + per_step - 1) / per_step * step_us[b] + 3.0) + (s > 0 ? 1.5 : 0.0);
      if (best == 0.0 || est < best) { best = est; BM = bms[b]; S = 1 << s; }
    }
  }
  if (BM == 32) return launch_cc_attn_bm<T, D, 32>(g, dev, q, k, v, cache, out, ws, S, pdl, st);
  if (BM == 16) return launch_cc_attn_bm<T, D, 16>(g, dev, q, k, v, cache, out, ws, S, pdl, st);
  return launch_cc_attn_bm<T, D, 8>(g, dev, q, k, v, cache, out, ws, S, pdl, st);
}
template <typename T, int D, int NK>
static cudaError_t launch_cc_score_nk(const Geom& g, int dev, const void* q, const void* k, void* cache, void* ws, bool pdl, cudaStream_t st) {
  constexpr int smem = kvc::score_cc_bytes<D, NK>();
  static bool attr_set[kMaxDevices] = {};
  if (cudaError_t e = opt_in_smem(kvc::score_cc_kernel<T, D, NK>, smem, attr_set, dev)) return e;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3((g.n_cand + NK - 1) / NK, g.Hkv, g.nl);
  lc.blockDim = dim3(kvc::kCcThreads, 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  LaunchAttrs la(0, pdl);
  lc.attrs = la.at;
  lc.numAttrs = la.n;
  return cudaLaunchKernelEx(&lc, kvc::score_cc_kernel<T, D, NK>, (const T*)q, (const T*)k, (const char*)cache, (char*)ws, g);
}
template <typename T, int D>
static cudaError_t launch_cc_score(const Geom& g, int dev, const void* q, const void* k, void* cache, void* ws, bool pdl, cudaStream_t st) {
  // 32 keys per CTA read the observer rows half as often (8 kv-heads x 608 keys, d = 64: 6.5 us against 7.5); 16 spread
  // a launch that does not fill the GPU over twice the SMs (2 x 1056 keys, d = 128: 7.9 us against 11.1)
  if ((long long)(g.n_cand + 31) / 32 * g.Hkv * g.nl > kvc::kNumSMs) return launch_cc_score_nk<T, D, 32>(g, dev, q, k, cache, ws, pdl, st);
  return launch_cc_score_nk<T, D, 16>(g, dev, q, k, cache, ws, pdl, st);
}

// Launch shape of the tensor-core attention: R row tiles per CTA (1 or 2) and, with one, the key split S over a cluster.
// The shapes are compared with a model of the kernel's duration.  It was fitted to device stamps of all five shapes on sixteen
// configurations while S still lay under P (us): a key tile cost 1.78 per pair of row tiles taking turns and 0.94 for a
// single tile (whose two softmax groups take alternate key tiles), a CTA 4.3 around them, the combine 2.7 (3.7 over eight CTAs); CTAs beyond
// what is resident at a time (one per SM; 32 clusters of four, 14 of eight) run as further waves.  Measured then, R=2 / R=1 S=1 /
// S=2 / S=4 / S=8:  196 x 4 rows, 8 kv-heads, 2244 keys 35.3 / 20.6 / 15.7 / 25.2 / 46.2;  576 x 7, 4, 1600 keys 28.2 /
// 17.0 / 27.3 / 45.9 / 92.9;  784 x 7, 4, 2832 keys 46.6 / 46.9 / 52.7;  1000 x 1, 32, 1500 keys 29.3 / 33.7 / 51.4;
// 256 x 4, 2, 1280 keys 21.3 / 12.9 / 10.9 / 9.3 / 18.1;  100 x 3, 4, 4100 keys 61.4 / 33.2 / 21.5 / 14.9 / 12.6;
// 128 x 1, 32, 320 keys 7.2 / 7.2 / 9.2 / 7.8 / 25.7.
// Since S has columns of its own a key tile costs 1.66 and 0.80, and the combine about 3.5.  Neither the figures above nor the
// constants have been taken again: with them some launches of three to six key tiles would not be split over four CTAs, and a
// last wave that is not full is charged as a full one.  (A changed shape groups a row's keys differently: the last bits of its
// log-sum-exp, and which of two candidates with scores that agree to seven digits is retained, may change with it.  Both are
// right; what has to be the same bits is a call with compress on a side stream and in stream order.)
// (An exchange of the partials through an L2-resident global buffer instead of distributed shared memory was measured
// too: slower, the release / acquire round trip costs more than the narrow SM-to-SM path.)
struct AttnShape { int R, S, n_pairs; long long ctas; };
static AttnShape attn_launch_shape(const Geom& g, bool allow_split, bool evict) {
  // SMs that mixed launches leave to a compress kernel on a side stream.  In stream order nobody needs them, but the
  // launch shape decides how a row's keys are grouped and thereby the last bits of the output: results must not depend on
  // KVC_FLAG_ASYNC_COMPRESS.  (In stream order this costs 4 - 6 % of a request whose launches are mixed, e.g. 784 x 7 rows
  // 1073 -> 1119 us; no reserve in either mode would cost 2 - 14 % on the side streams.)
  const int reserve = evict && g.nl == 1 ? std::min(4 * g.Hkv, kvc::kNumSMs) : 0;
  const int TOK = 128 / g.G;
  const int tiles = (g.n + TOK - 1) / TOK;
  const int Tc = (g.n_c + 127) / 128, T = Tc + (g.n + 127) / 128;
  const int capacity[4] = {kvc::kNumSMs, kvc::kNumSMs, 128, 112};
  const double combine_us[4] = {0.0, 2.7, 2.7, 3.7};
  const long long heads = (long long)g.Hkv * g.nl;
  auto waves = [](long long ctas, int cap) { return (double)((ctas + cap - 1) / cap); };
  AttnShape best = {2, 1, tiles / 2, (tiles - tiles / 2) * heads};
  double best_us = tiles == 1 ? INFINITY : waves(best.ctas, kvc::kNumSMs) * (T * 1.78 + 4.3);   // a single row tile never fills a pair
  // Pairs that would leave SMs idle: the row tiles with the most keys, the last ones, get a CTA each instead (1.2 us per
  // key tile there, measured with K and V tiles going round all four slots of their ring; now each kind has two).
  // 784 x 7 rows, 4 kv-heads, 2832 keys: 46.5 -> 38.2 us; 640 x 4, 8, d = 64 31.5 -> 25.7; 1024 x 4, 8, 5120 keys
  // 78.4 -> 76.6, all without the reserve.  With it, requests with compress on a side stream take, against none: 700 x 1 rows, 32 kv-heads 469 -> 411 us, 640 x 4, 8, d = 64 620 -> 604, 1024 x 4,
  // 8 2654 -> 2589, 784 x 7, 4 891 -> 898.
  const long long per_head = (kvc::kNumSMs - reserve) / heads;
  if (per_head > tiles - tiles / 2 && per_head < tiles) {
    const int n_pairs = (int)(tiles - per_head);
    const int T_pair = Tc + (std::min(g.n, 2 * n_pairs * TOK) + 127) / 128;
    const double est = std::max(T_pair * 1.78, T * 1.2) + 4.3;
    if (est < best_us) { best_us = est; best = {2, 1, n_pairs, (tiles - n_pairs) * heads}; }
  }
  for (int s = 0; s < (allow_split ? 4 : 1) && (1 << s) <= T; ++s) {
    const long long ctas = (tiles * heads) << s;
    double est = waves(ctas, capacity[s]) * ((T + (1 << s) - 1) / (1 << s) * 0.94 + 4.3) + combine_us[s];
    // A split that takes the last SMs a compress kernel on a side stream could run on must be worth that (whole calls, 32
    // kv-heads: 4 key tiles 13.2 us with S = 4 against 8.9 with S = 1; 11: 20.7 against 14.5 with S = 2; but 37 in stream order,
    // where the shape has to be the same, 37.4 against 43.9 with S = 2).
    if (s > 0 && evict && g.nl == 1 && ctas + heads > kvc::kNumSMs) est += 3.0;
    if (est < best_us) { best_us = est; best = {1, 1 << s, 0, ctas}; }
  }
  return best;
}

extern "C" int kvc_attention_shape(const kvc_ctx* c, int n, int n_c, int n_layers, int* row_tiles, int* key_split, int* pairs) {
  if (!live(c)) return KVC_ESTATE;
  if (!c->use_tc || n < 1 || n_c < 0 || n_layers < 1 || n_layers > c->cfg.n_layers || !row_tiles || !key_split || !pairs) return KVC_EINVAL;
  Geom g;
  memset(&g, 0, sizeof(g));
  g.n = n; g.n_c = n_c; g.G = c->G; g.Hkv = c->cfg.n_kv_heads; g.nl = n_layers;
  const AttnShape s = attn_launch_shape(g, !(c->cfg.flags & KVC_FLAG_NO_KEY_SPLIT), (long long)n_c + n > c->cfg.budget);
  *row_tiles = s.R; *key_split = s.S; *pairs = s.n_pairs;
  return KVC_OK;
}

template <int D, int R>
static cudaError_t launch_tc_attn(const Geom& g, int dev, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                  const CUtensorMap& tkin, const CUtensorMap& tvin, const CUtensorMap& tout, void* cache,
                                  void* out, void* ws, int S, int n_pairs, bool pdl, cudaStream_t st) {
  const int smem = (R + kvc::attn_stages<R>()) * (D / 64) * kvc::kSubTileBytes + 1024;
  static bool attr_set[kMaxDevices] = {};
  if (cudaError_t e = opt_in_smem(kvc::attn_tc_kernel<D, R>, smem, attr_set, dev)) return e;
  const int TOK = 128 / g.G;
  const int tiles = (g.n + TOK - 1) / TOK;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3(R == 1 ? tiles * S : tiles - n_pairs, g.Hkv, g.nl);
  lc.blockDim = dim3(kvc::kAttnThreads, 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  LaunchAttrs la(S, pdl);
  lc.attrs = la.at;
  lc.numAttrs = la.n;
  return cudaLaunchKernelEx(&lc, kvc::attn_tc_kernel<D, R>, tq, tk, tv, tkin, tvin, tout, (char*)cache, (__nv_bfloat16*)out,
                            (char*)ws, g, S, n_pairs);
}
// a2..a4 fused (compress.cuh).  MODE: kvc::kScoresGiven / kScoreAttention / kScoreKeyDiff.
template <int D, int MODE, int OBS = kvc::kMaxObsRowsFused>
static cudaError_t launch_compress(const Geom& g, int dev, const CUtensorMap& tk, const CUtensorMap& tqo, const CUtensorMap& tkin,
                                   const void* k, void* cache, void* ws, int elem_bytes, bool pdl, bool wide_ok, int cn_cap, cudaStream_t st) {
  const int score_bytes = MODE == kvc::kScoreAttention ? 2 * (D / 64) * kvc::kSubTileBytesC + (D / 64) * OBS * 128 : 0;
  const int table_bytes = kvc::kMaxKeysSmem * 8 + 2 * kvc::kMaxMovesSmem * 4 + 2 * kvc::kSelBins * 4;   // keys, move tables, histograms
  const int smem_min = (score_bytes > table_bytes ? score_bytes : table_bytes) + 1024;
  // More than half an SM: one CTA per SM.  With more than 128 observer rows that is a must: the CTA takes all of the SM's
  // TMEM, and CTAs of two clusters sharing SMs could each hold what the other's peer waits for.
  const int smem_solo = smem_min > 120 * 1024 ? smem_min : 120 * 1024;
  constexpr bool kAlone = OBS > kvc::kMaxObsRowsFused;
  static bool attr_set[kMaxDevices] = {};
  if (cudaError_t e = opt_in_smem(kvc::compress_kernel<D, MODE, OBS>, smem_solo, attr_set, dev)) return e;
  // Clusters of more than 8 CTAs are not portable: the kernel must allow them, and the device says how many clusters
  // of a size (one CTA per SM) it can hold at a time -- asked once per device and size; 0 where it refuses.
  static int wide_clusters[kMaxDevices][kvc::kMaxClusterWide + 1] = {};   // 0: not asked yet, -1: none, else clusters in flight
  auto clusters_in_flight = [&](int size) {
    int& slot = wide_clusters[dev][size];
    if (slot == 0) {
      int n_wide = 0;
      if (cudaFuncSetAttribute(kvc::compress_kernel<D, MODE, OBS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t q;
        memset(&q, 0, sizeof(q));
        q.gridDim = dim3(size, 1, 1);
        q.blockDim = dim3(kvc::kCompressThreads, 1, 1);
        q.dynamicSmemBytes = smem_solo;
        LaunchAttrs qa(size, false);
        q.attrs = qa.at;
        q.numAttrs = qa.n;
        if (cudaOccupancyMaxActiveClusters(&n_wide, kvc::compress_kernel<D, MODE, OBS>, &q) != cudaSuccess) n_wide = 0;
      }
      (void)cudaGetLastError();                           // a refusal is an answer, not an error of this call
      slot = n_wide > 0 ? n_wide : -1;
    }
    return slot;
  };
  // cluster size: spread one kv-head over several SMs when the heads alone cannot fill the GPU
  const int n_tiles = MODE == kvc::kScoreAttention ? (g.n_sc + 127) / 128 + (g.n_cand - g.n_sc + 127) / 128 : (g.n_cand + 127) / 128;
  int Cn = (int)(kvc::kNumSMs / ((long long)g.Hkv * g.nl));
  if (Cn > kvc::kMaxClusterWide) Cn = kvc::kMaxClusterWide;
  // More than the portable 8 CTAs only while every cluster of the launch can be resident at once, and only in stream
  // order: on a side stream the kernel shares the GPU with the next layer's attention, where a wider cluster waits
  // longer for its SMs than it saves (measured: the video workload's step went from 44 to 49 ms).
  if (!wide_ok && Cn > 8) Cn = 8;
  if (cn_cap > 0 && Cn > cn_cap) Cn = cn_cap;             // (side stream: stay within the SMs the attention leaves idle)
  while (Cn > 8 && clusters_in_flight(Cn) < (long long)g.Hkv * g.nl) --Cn;
  // One key tile per CTA in stream order while the launch stays small, else two: 2 kv-heads x 10 tiles 8.1 -> 7.6 us, 8 x 5 7.7 -> 7.3,
  // 8 x 18 9.7 -> 9.4; but 32 x 5 7.5 -> 7.7, 16 clusters of nine CTAs do not find their SMs at once (12.9 -> 24),
  // beside another attention (side stream) 32 x 3 1509 -> 1541 per request, and with 224 observer rows 1682 -> 1692.
  // (The query-agnostic score keeps two: the order of its sums depends on the cluster size.)
  const bool small = MODE == kvc::kScoreAttention && !kAlone && wide_ok && (long long)std::min(Cn, n_tiles) * g.Hkv * g.nl <= 100;
  const int tiles_per_cta = small ? 1 : 2;                // fewer, and the cluster barriers cost more than the tiles
  if (Cn > (n_tiles + tiles_per_cta - 1) / tiles_per_cta) Cn = (n_tiles + tiles_per_cta - 1) / tiles_per_cta;
  // Clusters that the GPU cannot hold at once (one CTA per SM: 15 of seven to nine, 22 of six, 33 of four) run in two waves:
  // 16 kv-heads x 12 key tiles 30.1 -> 24.2 us per call with clusters of six for seven, 24 x 32 46.3 -> 34.1 with five for six.
  if (MODE != kvc::kScoreKeyDiff)
    while (Cn > 1 && (long long)Cn * g.Hkv * g.nl <= kvc::kNumSMs && clusters_in_flight(Cn) < (long long)g.Hkv * g.nl) --Cn;
  if (Cn < 1) Cn = 1;
  // Two CTAs share an SM only when there are more CTAs than SMs (then one scores while the other selects);
  // a launch that fits the GPU asks for more than half an SM's shared memory so that every CTA gets an SM
  // of its own instead of being packed in pairs.
  const int smem = !kAlone && (long long)Cn * g.Hkv * g.nl > kvc::kNumSMs ? smem_min : smem_solo;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3(Cn, g.Hkv, g.nl);
  lc.blockDim = dim3(kvc::kCompressThreads, 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  LaunchAttrs la(Cn, pdl);
  lc.attrs = la.at;
  lc.numAttrs = la.n;
  return cudaLaunchKernelEx(&lc, kvc::compress_kernel<D, MODE, OBS>, tk, tqo, tkin, (const char*)k, (char*)cache, (char*)ws, g, Cn, elem_bytes);
}

template <int D>
static cudaError_t launch_tc_score(const Geom& g, int dev, const CUtensorMap& tk, const CUtensorMap& tqo, void* ws,
                                   int tok_per_group, cudaStream_t st) {
  const int smem = (D / 64) * (kvc::kSubTileBytes + 256 * 128) + 1024;
  static bool attr_set[kMaxDevices] = {};
  if (cudaError_t e = opt_in_smem(kvc::score_tc_kernel<D>, smem, attr_set, dev)) return e;
  dim3 grid((g.n_cand + 127) / 128, g.Hkv, g.nl);
  kvc::score_tc_kernel<D><<<grid, 128, smem, st>>>(tk, tqo, (char*)ws, g, tok_per_group);
  return cudaSuccess;
}

static int run_chunk(kvc_ctx* c, int layer0, int nl, const void* q, long long q_ls, const void* k, const void* v,
                     long long kv_ls, int n, long long pos0, void* cache, size_t cache_ls, void* ws, void* out,
                     long long out_ls, cudaStream_t st, int n_proxy = 0, bool allow_async = true,
                     bool clear_status = false) {
  const kvc_config& cf = c->cfg;
  if (layer0 < 0 || nl < 1 || layer0 + nl > cf.n_layers) return fail(c, KVC_EINVAL, "layer range [%d, %d) outside [0, %d)", layer0, layer0 + nl, cf.n_layers);
  if (!q || !k || !v || !cache || !ws || !out) return fail(c, KVC_EINVAL, "null pointer argument");
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(cache) || !aligned16(ws) || !aligned16(out))
    return fail(c, KVC_EINVAL, "pointers must be 16-byte aligned");
  // Blocks hold at most max_chunk tokens, except that an EMPTY cache may be filled with up to B tokens in one
  // pass (hybrid schedule, Sec. 5, Budgeting: the first M tokens go through in a single forward): nothing is evicted then.
  const int n_limit = (c->len[layer0] == 0 && cf.budget > cf.max_chunk) ? cf.budget : cf.max_chunk;
  if (n < 1 || n > n_limit) return fail(c, KVC_EINVAL, "n = %d outside [1, %d] (max_chunk = %d; up to B = %d into an empty cache)", n, n_limit, cf.max_chunk, cf.budget);
  if (pos0 < 0 || pos0 + n > 0x7fffffffLL) return fail(c, KVC_EINVAL, "pos0 out of range");
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != cf.device)
    return fail(c, KVC_ESTATE, "current CUDA device %d is not the context's device %d", dev, cf.device);
  const int n_c = c->len[layer0];
  for (int i = 0; i < nl; ++i) {
    if (c->len[layer0 + i] < 0) return fail(c, KVC_ESTATE, "layer %d used before kvc_reset", layer0 + i);
    if (c->len[layer0 + i] != n_c) return fail(c, KVC_ESTATE, "batched layers hold different cache lengths");
  }
  if (nl > 1) {
    const long long qmin = (long long)n * cf.n_q_heads * cf.head_dim, kmin = (long long)n * cf.n_kv_heads * cf.head_dim;
    if (q_ls < qmin || out_ls < qmin || kv_ls < kmin || cache_ls < c->blob_bytes)
      return fail(c, KVC_EINVAL, "layer strides too small");
    if ((q_ls * c->elem) % 16 || (out_ls * c->elem) % 16 || (kv_ls * c->elem) % 16 || cache_ls % 16)
      return fail(c, KVC_EINVAL, "layer strides must be multiples of 16 bytes");
  } else {
    q_ls = out_ls = (long long)n * cf.n_q_heads * cf.head_dim;
    kv_ls = (long long)n * cf.n_kv_heads * cf.head_dim;
    cache_ls = c->blob_bytes;
  }

  Geom g;
  memset(&g, 0, sizeof(g));
  if (n_proxy < 0 || n_proxy >= n) return fail(c, KVC_EINVAL, "n_proxy = %d outside [0, n = %d)", n_proxy, n);
  // Proxy query tokens (the last n_proxy rows) are appended and attended like the rest of the block, but
  // the cache ends before them: rows tot .. tot + n_proxy are left behind as unused space, the proxies
  // are the observers, and with no protected window every entry competes for the B places.
  g.n = n; g.n_c = n_c; g.tot = n_c + n - n_proxy; g.B = cf.budget;
  g.w = n_proxy ? n_proxy : (c->w_cfg < n ? c->w_cfg : n);
  g.G = c->G; g.Hq = cf.n_q_heads; g.Hkv = cf.n_kv_heads; g.d = cf.head_dim; g.cap = c->cap; g.nl = nl;
  g.max_chunk = cf.max_chunk;
  g.n_cand = n_proxy ? g.tot : g.tot - g.w;
  g.n_keep = n_proxy ? g.B : g.B - g.w;
  g.scale_log2 = c->scale * 1.4426950408889634f;
  g.pos0 = pos0;
  g.q_ls = q_ls; g.kv_ls = kv_ls; g.out_ls = out_ls; g.cache_ls = (long long)cache_ls;
  g.v_off = (long long)c->v_off; g.pos_off = (long long)c->pos_off;
  g.ws_ls = (long long)c->ws_slot_bytes;
  // KVC_FLAG_ASYNC_COMPRESS: score / select / compact of a layer run on a side stream, beside whatever the caller
  // enqueues next (the next layer's attention, in a decoder stack, needs this layer's output, not its compacted
  // cache); the layer then works in its own workspace slot, and the next call that touches the layer waits
  const bool async_compress = (cf.flags & 16u) && nl == 1 && allow_async && c->use_tc;
  g.slot0 = async_compress ? layer0 : 0;
  // In stream order the score phase reads the block's keys from the input and so can start before the attention has
  // ended; on a side stream the caller may reuse k by then.
  g.n_sc = async_compress ? g.tot : g.n_c;
  if (g.n_sc > g.n_cand && cf.policy != KVC_SCORE_KEYDIFF) g.n_sc = g.n_cand;
  g.lse_off = c->lse_off; g.score_off = c->score_off; g.msrc_off = c->msrc_off; g.mdst_off = c->mdst_off;
  g.mcount_off = c->mcount_off;
  g.wait_limit_k = c->wait_limit_k;
  const bool evict = g.tot > g.B;                      // Alg. 1: "if |C| > M"
  const bool f32 = cf.dtype == KVC_F32;
  const int D = cf.head_dim;

  // tensor maps first: nothing is enqueued if an encode fails
  CUtensorMap tq, tk, tv, tqo, tkin, tvin, tout;
  int tok_per_group = 0;
  if (c->use_tc) {
    int rc = get_encoder(c);
    if (rc) return rc;
    const int TOK = 128 / g.G;
    const uint64_t qd[4] = {(uint64_t)D, (uint64_t)g.Hq, (uint64_t)n, (uint64_t)nl};
    const uint64_t qs[3] = {(uint64_t)D * 2, (uint64_t)g.Hq * D * 2, (uint64_t)q_ls * 2};
    const uint32_t qb[4] = {64, (uint32_t)g.G, (uint32_t)TOK, 1};
    if ((rc = make_map(c, &tq, q, qd, qs, qb))) return rc;
    const uint64_t os[3] = {(uint64_t)D * 2, (uint64_t)g.Hq * D * 2, (uint64_t)out_ls * 2};
    if ((rc = make_map(c, &tout, out, qd, os, qb))) return rc;
    const uint64_t kd[4] = {(uint64_t)D, (uint64_t)g.cap, (uint64_t)g.Hkv, (uint64_t)nl};
    const uint64_t ks[3] = {(uint64_t)D * 2, (uint64_t)g.cap * D * 2, (uint64_t)cache_ls};
    const uint32_t kb[4] = {64, 128, 1, 1};
    if ((rc = make_map(c, &tk, cache, kd, ks, kb))) return rc;
    if ((rc = make_map(c, &tv, (char*)cache + c->v_off, kd, ks, kb))) return rc;
    // the block's own keys / values, read in place: k, v are [n][Hkv][d]
    const uint64_t id[4] = {(uint64_t)D, (uint64_t)g.Hkv, (uint64_t)n, (uint64_t)nl};
    const uint64_t is[3] = {(uint64_t)D * 2, (uint64_t)g.Hkv * D * 2, (uint64_t)kv_ls * 2};
    const uint32_t ib[4] = {64, 1, 128, 1};
    if ((rc = make_map(c, &tkin, k, id, is, ib))) return rc;
    if ((rc = make_map(c, &tvin, v, id, is, ib))) return rc;
    if (evict) {
      tok_per_group = 256 / g.G;
      if (tok_per_group > g.w) tok_per_group = g.w;
      const uint32_t ob[4] = {64, (uint32_t)g.G, (uint32_t)tok_per_group, 1};
      if ((rc = make_map(c, &tqo, q, qd, qs, ob))) return rc;
    }
  }

  const bool pdl_main = !(cf.flags & 8u);              // flag 8: plain stream order between the kernels (diagnostic)
  const bool pdl = pdl_main;
  cudaError_t e = cudaSuccess;
  if (int rc = wait_pending(c, layer0, layer0 + nl, st)) return rc;    // a compress kernel of an earlier block may still run
  // ... and one of another layer in a workspace slot of this call: a single-layer call with compress on the side stream works
  // in its layer's slot, a batched call and kvc_prefill_chunk_host in the first ones (the built-in scratch is not shared so)
  if (!clear_status)
    if (int rc = wait_slots(c, g.slot0, g.slot0 + nl, st)) return rc;
  // every host check has passed: from here on work is enqueued.  A workspace that keeps an earlier user's contents
  // (the built-in scratch array) gets its status word cleared first.
  if (clear_status)
    if (int rc = check_cuda(c, cudaMemsetAsync(ws, 0, kvc::kWsHeaderBytes, st), "cudaMemsetAsync(status word)")) return rc;
  // a0 append + a1 attention
  long long attn_ctas = 0;                                    // CTAs of the attention launch (tensor-core path)
  {
  ProfScope ps(c, 1, st);
  g.stamps = next_stamp(c, 1);
  if (c->use_tc) {
    const AttnShape sh = attn_launch_shape(g, !(cf.flags & 4u), evict);
    attn_ctas = sh.ctas;
    // The query-agnostic kernel needs nothing of the attention up to its moves: it starts at once if it fits beside it.  Us
    // per request, started at once / at the end of the key loop (CTAs of attention + compress): 88 + 32 1281 / 1672, 32 + 64
    // 2381 / 2962, 112 + 20 2112 / 2641, 72 + 16 677 / 892.  Without room it costs beside an attention that is short or splits its
    // keys (112 + 40 3258 / 3191, 112 + 72 4855 / 4787, 88 + 64 2388 / 2379, 64 + 128 1346 / 1338); beside a long one that does
    // not it would gain (128 + 28 1124 / 1171 with the blocks that fit started at once, 128 + 128 2718 / 2812, 132 + 44 1367 /
    // 1577).  The query-aware kernel has only loads and products to do early, for which the end of the key loop is soon enough.
    const long long heads = (long long)g.Hkv * g.nl;
    const long long cluster = std::min<long long>({kvc::kMaxClusterWide, kvc::kNumSMs / heads, (g.n_cand + 255) / 256});
    g.early = evict && !async_compress && cf.policy == KVC_SCORE_KEYDIFF && cluster > 0 && attn_ctas + heads * cluster <= kvc::kNumSMs;
    auto launch = [&](auto launcher) { return launcher(g, dev, tq, tk, tv, tkin, tvin, tout, cache, out, ws, sh.S, sh.n_pairs, pdl, st); };
    if (D == 128) e = sh.R == 2 ? launch(launch_tc_attn<128, 2>) : launch(launch_tc_attn<128, 1>);
    else e = sh.R == 2 ? launch(launch_tc_attn<64, 2>) : launch(launch_tc_attn<64, 1>);
  } else {
    auto launch = [&](auto launcher) { return launcher(g, dev, q, k, v, cache, out, ws, !(cf.flags & 4u), pdl, st); };
    if (f32) e = D == 128 ? launch(launch_cc_attn<float, 128>) : launch(launch_cc_attn<float, 64>);
    else e = D == 128 ? launch(launch_cc_attn<__nv_bfloat16, 128>) : launch(launch_cc_attn<__nv_bfloat16, 64>);
  }
  }
  if (e != cudaSuccess) return check_cuda(c, e, "attention launch setup");
  c->launches++;
  if (evict) {
    if (async_compress) {
      if (int rc = ensure_side_stream(c)) return rc;
      if ((e = cudaEventRecord(c->ev_attn[layer0], st)) != cudaSuccess || (e = cudaStreamWaitEvent(c->side[layer0 % kvc_ctx::kSideStreams], c->ev_attn[layer0], 0)) != cudaSuccess)
        return check_cuda(c, e, "side stream fork");
      st = c->side[layer0 % kvc_ctx::kSideStreams];                                           // everything below goes to the side stream
    }
    const bool pdl = pdl_main && !async_compress;             // an event, not a kernel, precedes the side stream's launches
    g.stamp_early = !pdl;
    // On a side stream the kernel runs beside the next layer's attention, a launch of the same shape as this
    // layer's: a cluster per kv-head that fits the SMs that launch leaves idle shares nothing with it, while a wider
    // one takes SMs from attention CTAs, which then start late and lengthen the launch everything else waits for
    // (measured on the video workload: 44.3 -> 39.5 ms per step).
    int cn_cap = 0;
    if (async_compress && attn_ctas > 0 && kvc::kNumSMs - attn_ctas >= (long long)g.Hkv * g.nl) {
      const long long idle = kvc::kNumSMs - attn_ctas;
      cn_cap = (int)(idle / ((long long)g.Hkv * g.nl));
      // ... and a cluster must find its SMs inside one GPC, where the attention leaves about idle / 8 of them: a
      // cluster larger than that waits for attention CTAs to leave (tiled-image workload, 20 idle SMs, 4 kv-heads:
      // clusters of 4 or 5 CTAs 2.69e7 tokens/s/layer, of 3 or fewer 2.79e7).
      const int per_gpc = (int)((idle + 4) / 8);
      if (cn_cap > per_gpc) cn_cap = per_gpc > 0 ? per_gpc : 1;
    }
    const bool keydiff = cf.policy == KVC_SCORE_KEYDIFF;      // query-agnostic: always scored inside the fused kernel
    // Up to 128 observer rows are scored inside the fused kernel too, up to 256 with the CTA alone on its SM: that saves
    // the score kernel's launch and start-up (4 kv-heads x 2300 keys x 224 rows, in stream order: 12.3 us against 5.0 + 8.0
    // and 1.5 between them; 16 x 1250 x 256: 12.9 against 6.7 + 7.9).  Exception: two such launches in flight on the side
    // streams that would not both fit the SMs the attention leaves idle (8 kv-heads, 20 idle SMs: 4 % of a step slower).
    const bool wide_obs = g.w * g.G > kvc::kMaxObsRowsFused;
    const long long side_ctas = 2ll * g.Hkv * g.nl * std::min(cn_cap, (int)((g.n_cand + 255) / 256));
    const bool crowded = cn_cap > 0 && side_ctas > kvc::kNumSMs - attn_ctas;
    const bool fused_score = !keydiff && c->use_tc && g.w * g.G <= (crowded ? kvc::kMaxObsRowsFused : kvc::kMaxObsRowsWide);
    if (!fused_score && !keydiff) {
      // a2 score as a kernel of its own (fp32 on CUDA cores; bf16 with more observer rows per kv-head than the fused
      // kernel takes)
      ProfScope ps(c, 2, st);
      g.stamps = next_stamp(c, 2);
      if (c->use_tc) {
        e = D == 128 ? launch_tc_score<128>(g, dev, tk, tqo, ws, tok_per_group, st) : launch_tc_score<64>(g, dev, tk, tqo, ws, tok_per_group, st);
      } else if (f32) {
        e = D == 128 ? launch_cc_score<float, 128>(g, dev, q, k, cache, ws, pdl, st) : launch_cc_score<float, 64>(g, dev, q, k, cache, ws, pdl, st);
      } else {
        e = D == 128 ? launch_cc_score<__nv_bfloat16, 128>(g, dev, q, k, cache, ws, pdl, st) : launch_cc_score<__nv_bfloat16, 64>(g, dev, q, k, cache, ws, pdl, st);
      }
      if (e != cudaSuccess) return check_cuda(c, e, "score launch");
      c->launches++;
    }
    // (a2 +) a3 select + a4 compact
    {
      ProfScope ps(c, 3, st);
      g.stamps = next_stamp(c, 3);
      if (keydiff) e = launch_compress<64, kvc::kScoreKeyDiff>(g, dev, tk, tk, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st);
      else if (fused_score && wide_obs)
        e = D == 128 ? launch_compress<128, kvc::kScoreAttention, kvc::kMaxObsRowsWide>(g, dev, tk, tqo, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st)
                     : launch_compress<64, kvc::kScoreAttention, kvc::kMaxObsRowsWide>(g, dev, tk, tqo, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st);
      else if (fused_score) e = D == 128 ? launch_compress<128, kvc::kScoreAttention>(g, dev, tk, tqo, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st)
                                         : launch_compress<64, kvc::kScoreAttention>(g, dev, tk, tqo, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st);
      else e = launch_compress<64, kvc::kScoresGiven>(g, dev, tk, tk, tkin, k, cache, ws, (int)c->elem, pdl, !async_compress, cn_cap, st);
    }
    if (e != cudaSuccess) return check_cuda(c, e, "compress launch");
    c->launches++;
    if (async_compress) {
      if ((e = cudaEventRecord(c->ev_comp[layer0], st)) != cudaSuccess) return check_cuda(c, e, "side stream event");
      c->pending[layer0] = 1;
    }
  }
  int rc = check_cuda(c, cudaGetLastError(), "kernel launch");
  if (rc) return rc;
  const int new_len = evict ? g.B : g.tot;
  for (int i = 0; i < nl; ++i) c->len[layer0 + i] = new_len;
  return KVC_OK;
}

extern "C" int kvc_prefill_chunk(kvc_ctx* c, int layer, const void* q, const void* k, const void* v, int n,
                                 long long pos0, void* cache, void* workspace, void* out, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  return run_chunk(c, layer, 1, q, 0, k, v, 0, n, pos0, cache, 0, workspace, out, 0, (cudaStream_t)stream);
}

extern "C" int kvc_prefill_chunk_proxy(kvc_ctx* c, int layer, const void* q, const void* k, const void* v, int n,
                                       int n_proxy, long long pos0, void* cache, void* workspace, void* out, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (n_proxy < 1) return fail(c, KVC_EINVAL, "n_proxy = %d: at least one proxy token is needed (use kvc_prefill_chunk otherwise)", n_proxy);
  return run_chunk(c, layer, 1, q, 0, k, v, 0, n, pos0, cache, 0, workspace, out, 0, (cudaStream_t)stream, n_proxy);
}

extern "C" int kvc_prefill_chunk_layers(kvc_ctx* c, int layer0, int n_layers, const void* q, long long q_layer_stride,
                                        const void* k, const void* v, long long kv_layer_stride, int n, long long pos0,
                                        void* cache, size_t cache_layer_stride, void* workspace, void* out,
                                        long long out_layer_stride, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  return run_chunk(c, layer0, n_layers, q, q_layer_stride, k, v, kv_layer_stride, n, pos0, cache, cache_layer_stride,
                   workspace, out, out_layer_stride, (cudaStream_t)stream);
}

// q, k, v and out of one block, each rounded up to 256 bytes
static size_t staging_half_bytes(size_t qb, size_t kb) { return 2 * align_up(qb, 256) + 2 * align_up(kb, 256); }

extern "C" int kvc_staging_nbytes(const kvc_ctx* c, size_t* nbytes) {
  if (!live(c)) return KVC_ESTATE;
  if (!nbytes) return KVC_EINVAL;
  const size_t rows = c->cfg.max_chunk > c->cfg.budget ? c->cfg.max_chunk : c->cfg.budget;   // room for a bulk first block
  const size_t qb = rows * c->cfg.n_q_heads * c->cfg.head_dim * c->elem;
  const size_t kb = rows * c->cfg.n_kv_heads * c->cfg.head_dim * c->elem;
  *nbytes = 2 * staging_half_bytes(qb, kb);                  // two halves: the copies of one block run beside the previous block
  return KVC_OK;
}

static int ensure_copy_stream(kvc_ctx* c) {
  if (c->copy_in) return KVC_OK;                             // set last: marks a complete set
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
    if (!c->ev_in[i] && (e = cudaEventCreateWithFlags(&c->ev_in[i], cudaEventDisableTiming)) != cudaSuccess) c->ev_in[i] = nullptr;
    if (e == cudaSuccess && !c->ev_free[i] && (e = cudaEventCreateWithFlags(&c->ev_free[i], cudaEventDisableTiming)) != cudaSuccess) c->ev_free[i] = nullptr;
    if (e == cudaSuccess && !c->ev_out[i] && (e = cudaEventCreateWithFlags(&c->ev_out[i], cudaEventDisableTiming)) != cudaSuccess) c->ev_out[i] = nullptr;
  }
  if (e != cudaSuccess) return fail(c, KVC_ECUDA, "cudaEventCreate: %s", cudaGetErrorString(e));
  if (!c->copy_out && (e = cudaStreamCreateWithFlags(&c->copy_out, cudaStreamNonBlocking)) != cudaSuccess) {
    c->copy_out = nullptr;
    return fail(c, KVC_ECUDA, "cudaStreamCreate: %s", cudaGetErrorString(e));
  }
  if ((e = cudaStreamCreateWithFlags(&c->copy_in, cudaStreamNonBlocking)) != cudaSuccess) {
    c->copy_in = nullptr;
    return fail(c, KVC_ECUDA, "cudaStreamCreate: %s", cudaGetErrorString(e));
  }
  return KVC_OK;
}

extern "C" int kvc_prefill_chunk_host(kvc_ctx* c, int layer, const void* q_host, const void* k_host, const void* v_host,
                                      int n, long long pos0, void* cache, void* workspace, void* staging, void* out_host,
                                      void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (!q_host || !k_host || !v_host || !out_host || !staging) return fail(c, KVC_EINVAL, "null pointer argument");
  if (layer < 0 || layer >= c->cfg.n_layers) return fail(c, KVC_EINVAL, "layer %d outside [0, %d)", layer, c->cfg.n_layers);
  const int n_limit = (c->len[layer] == 0 && c->cfg.budget > c->cfg.max_chunk) ? c->cfg.budget : c->cfg.max_chunk;
  if (n < 1 || n > n_limit) return fail(c, KVC_EINVAL, "n = %d outside [1, %d]", n, n_limit);
  if (!aligned16(staging)) return fail(c, KVC_EINVAL, "staging must be 16-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  const size_t qb = (size_t)n * c->cfg.n_q_heads * c->cfg.head_dim * c->elem;
  const size_t kb = (size_t)n * c->cfg.n_kv_heads * c->cfg.head_dim * c->elem;
  size_t total = 0;
  kvc_staging_nbytes(c, &total);
  int rc = ensure_copy_stream(c);
  if (rc) return rc;
  // Calls alternate between the two halves of the staging buffer.  The inputs travel on the context's inbound copy
  // stream, behind the block that last read this half (two calls ago); the caller's stream waits for them and runs
  // the block; `out` goes back on the context's outbound copy stream, behind the block.  So the inbound copies of
  // call i+1, the kernels of call i+1 (other half) and the outbound copy of call i all run at the same time.  The
  // caller's stream then waits for the outbound copy of the PREVIOUS call (the other half: its `out` area is the
  // next block's), which has had this call's kernels to finish.
  const int half = (int)(c->host_calls & 1u);
  // The areas of a half start where those of the largest block do, whatever n is: the inbound copies of a call may run
  // while `out` of the call two before it, in the same half, is still on its way out.
  const size_t rows = c->cfg.max_chunk > c->cfg.budget ? c->cfg.max_chunk : c->cfg.budget;
  const size_t q_area = align_up(rows * c->cfg.n_q_heads * c->cfg.head_dim * c->elem, 256);
  const size_t k_area = align_up(rows * c->cfg.n_kv_heads * c->cfg.head_dim * c->elem, 256);
  char* dq = (char*)staging + half * (total / 2);
  char* dk = dq + q_area;
  char* dv = dk + k_area;
  char* dout = dv + k_area;
  if ((rc = check_cuda(c, cudaStreamWaitEvent(c->copy_in, c->ev_free[half], 0), "cudaStreamWaitEvent"))) return rc;
  if ((rc = check_cuda(c, cudaMemcpyAsync(dq, q_host, qb, cudaMemcpyHostToDevice, c->copy_in), "H2D q"))) return rc;
  if ((rc = check_cuda(c, cudaMemcpyAsync(dk, k_host, kb, cudaMemcpyHostToDevice, c->copy_in), "H2D k"))) return rc;
  if ((rc = check_cuda(c, cudaMemcpyAsync(dv, v_host, kb, cudaMemcpyHostToDevice, c->copy_in), "H2D v"))) return rc;
  if ((rc = check_cuda(c, cudaEventRecord(c->ev_in[half], c->copy_in), "cudaEventRecord"))) return rc;
  if ((rc = check_cuda(c, cudaStreamWaitEvent(st, c->ev_in[half], 0), "cudaStreamWaitEvent"))) return rc;
  rc = run_chunk(c, layer, 1, dq, 0, dk, dv, 0, n, pos0, cache, 0, workspace, dout, 0, st, 0, false);   // staging is reused: no side stream
  if (rc) return rc;
  c->host_calls++;                                           // (a rejected call leaves its half to the next one)
  if ((rc = check_cuda(c, cudaEventRecord(c->ev_free[half], st), "cudaEventRecord"))) return rc;
  if ((rc = check_cuda(c, cudaStreamWaitEvent(c->copy_out, c->ev_free[half], 0), "cudaStreamWaitEvent"))) return rc;
  if ((rc = check_cuda(c, cudaMemcpyAsync(out_host, dout, qb, cudaMemcpyDeviceToHost, c->copy_out), "D2H out"))) return rc;
  if ((rc = check_cuda(c, cudaEventRecord(c->ev_out[half], c->copy_out), "cudaEventRecord"))) return rc;
  // (an event that was never recorded counts as complete: the first call waits for nothing here)
  return check_cuda(c, cudaStreamWaitEvent(st, c->ev_out[1 - half], 0), "cudaStreamWaitEvent");
}

extern "C" int kvc_host_flush(kvc_ctx* c, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (!c->copy_out) return KVC_OK;                           // no host call yet
  for (int i = 0; i < 2; ++i)
    if (int rc = check_cuda(c, cudaStreamWaitEvent((cudaStream_t)stream, c->ev_out[i], 0), "cudaStreamWaitEvent")) return rc;
  return KVC_OK;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free variant: the scratch area is a fixed device array compiled into the library.
// In host code `g_static_ws` is only a handle for the runtime, not a device address; the address
// each device gives it is looked up once per device and cached here.
static __device__ __align__(256) unsigned char g_static_ws[KVC_STATIC_WS_BYTES];
static void* g_static_ws_ptr[kMaxDevices] = {nullptr};

static int static_ws_for_current_device(kvc_ctx* c, void** ptr) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return check_cuda(c, e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(c, KVC_EINVAL, "device ordinal %d not supported by the static scratch", dev);
  if (dev != c->cfg.device) return fail(c, KVC_ESTATE, "current CUDA device %d is not the context's device %d", dev, c->cfg.device);
  if (!g_static_ws_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_ws);
    if (e != cudaSuccess || !p) return check_cuda(c, e == cudaSuccess ? cudaErrorInvalidSymbol : e, "cudaGetSymbolAddress(static scratch)");
    g_static_ws_ptr[dev] = p;
  }
  *ptr = g_static_ws_ptr[dev];
  return KVC_OK;
}

extern "C" int kvc_prefill_chunk_static(kvc_ctx* c, int layer, const void* q, const void* k, const void* v, int n,
                                        long long pos0, void* cache, void* out, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  if (c->profiling) return fail(c, KVC_ESTATE, "kvc_prefill_chunk_static needs profiling off");
  const size_t need = kvc::kWsHeaderBytes + c->ws_slot_bytes;          // header + one layer slot
  if (need > (size_t)KVC_STATIC_WS_BYTES)
    return fail(c, KVC_EINVAL, "configuration needs %zu bytes of scratch, the built-in scratch holds %u", need,
                (unsigned)KVC_STATIC_WS_BYTES);
  void* ws = nullptr;
  int rc = static_ws_for_current_device(c, &ws);
  if (rc) return rc;
  // the array keeps the previous call's contents: only the status word has to start at zero, and it is cleared
  // once the argument and state checks have passed (a rejected call enqueues nothing)
  return run_chunk(c, layer, 1, q, 0, k, v, 0, n, pos0, cache, 0, ws, out, 0, (cudaStream_t)stream, 0, false, true);
}

extern "C" int kvc_status_static(kvc_ctx* c, void* stream) {
  if (!live(c)) return KVC_ESTATE;
  void* ws = nullptr;
  int rc = static_ws_for_current_device(c, &ws);
  if (rc) return rc;
  return kvc_status(c, ws, stream);
}
