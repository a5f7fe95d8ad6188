// One CTA of the kernel named on the command line, in the emulator: key=value arguments, lists as index:ms,index:ms
#include "emu.h"
#include <sstream>
#include "kernels.h"   // the kernels' sources as they are, without their includes

alignas(1024) uint8_t emu_smem[256 * 1024];
namespace kvc { uint8_t* smem_raw = emu_smem; }

static std::map<std::string, std::string> args;
static int num(const char* key, int other) { return args.count(key) ? atoi(args[key].c_str()) : other; }
static std::map<int, int> pairs(const char* key) {
  std::map<int, int> m;
  std::stringstream ss(args[key]);
  for (std::string item; std::getline(ss, item, ',');) m[atoi(item.c_str())] = atoi(item.c_str() + item.find(':') + 1);
  return m;
}

int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const std::string a = argv[i];
    args[a.substr(0, a.find('='))] = a.substr(a.find('=') + 1);
  }
  emu::load_ms = pairs("load_ms");
  emu::suspend_ms = pairs("suspend_ms");
  emu::mma_us = num("mma_us", 20);
  emu::pdl_ms = num("pdl_ms", 0);
  emu::copy_ms = num("copy_ms", 1);
  emu::load_parts = 1;                                     // d = 64: one box per tile
  const int S = num("split", 1), R = num("row_tiles", 1);
  kvc::Geom g;
  memset(&g, 0, sizeof(g));
  g.n = num("n", 128); g.n_c = num("n_c", 128); g.tot = g.n + g.n_c; g.B = num("budget", 1 << 20); g.w = num("w", 8);
  g.G = g.Hq = 1; g.d = 64; g.nl = 1; g.cap = 4096; g.max_chunk = 512;
  g.n_cand = g.tot - g.w; g.n_keep = g.B - g.w; g.n_sc = g.n_c;
  g.scale_log2 = 1.f;
  g.q_ls = g.kv_ls = g.out_ls = 64 * 512;
  g.v_off = 64ll * 2 * g.cap; g.pos_off = 2 * g.v_off; g.cache_ls = g.pos_off + 4 * g.cap;
  g.score_off = 4 * g.max_chunk; g.msrc_off = g.score_off + 4 * g.cap; g.mdst_off = g.msrc_off + 4 * g.max_chunk;
  g.mcount_off = g.mdst_off + 4 * g.max_chunk; g.ws_ls = g.mcount_off + 256;
  g.wait_limit_k = num("limit_ms", 20) * 1000000 / 1024;   // (a clock of the emulator: a nanosecond)
  std::vector<char> cache(g.cache_ls + 256), ws(kvc::kWsHeaderBytes + g.ws_ls);
  std::vector<__nv_bfloat16> out(64 * 512);
  for (int i = 0; i < g.tot; ++i) reinterpret_cast<int*>(cache.data() + g.pos_off)[i] = i;
  CUtensorMap tm;
  memset(&tm, 0, sizeof(tm));
  const int n_pairs = R == 2 ? 1 : 0;
  int rc = 2;
  if (args["kernel"] == "attention") {
    emu::grid_dim.x = R == 1 ? (g.n + 127) / 128 * S : (g.n + 127) / 128 - n_pairs;
    emu::copies_due = S > 1;
    auto call = [&](auto kernel) { return emu::run(kvc::kAttnThreads, [&, kernel] { kernel(tm, tm, tm, tm, tm, tm, cache.data(), out.data(), ws.data(), g, S, n_pairs); }); };
    // (without a key split the CTA with the lowest index has the last row tile: the pair is the last of two CTAs)
    if (R == 2) emu::block_idx.x = emu::grid_dim.x - 1;
    rc = R == 1 ? call(kvc::attn_tc_kernel<64, 1>) : call(kvc::attn_tc_kernel<64, 2>);
  }
  if (args["kernel"] == "compress")
    rc = emu::run(kvc::kCompressThreads, [&] { kvc::compress_kernel<64, kvc::kScoreAttention, 128>(tm, tm, tm, nullptr, cache.data(), ws.data(), g, 1, 2); });
  if (args["kernel"] == "score")
    rc = emu::run(128, [&] { kvc::score_tc_kernel<64>(tm, tm, ws.data(), g, 256); });
  printf("status %d\n", *reinterpret_cast<int*>(ws.data()));
  return rc;
}
