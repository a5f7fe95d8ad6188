"""GPU tests of the corners around the hot path: the query-agnostic score on degenerate keys (Sec. 3.2: keys
parallel to the anchor, identical keys, a zero key), the bounded device-side wait running out, and the guard
regions that the parity helper keeps around every buffer."""
import ctypes

import numpy as np
import pytest
import torch

from oracle.kvc_oracle import KVCOracle
from paper_2604_16734_b200 import binding
from paper_2604_16734_b200.binding import Kvc, KVC_ETIMEOUT, KVC_FLAG_ASYNC_COMPRESS

from parity_util import check_guards, compare_chunk, guarded_copy, install_guards

pytestmark = pytest.mark.gpu


# ------------------------------------------------------------------------------------------------
# query-agnostic score (Sec. 3.2) where the cosine reaches 1: the keys the policy must evict first

def _parallel_keys(a, n, specials):
    """n keys per kv-head that are all positive power-of-two multiples of the direction a ([1][Hkv][d]; so every
    cosine to the anchor is exactly the same number in any precision), except the rows named in `specials`:
    'neg' = -a (the least similar key there can be), 'neg2' = -2a, 'zero' = the zero key."""
    scale = torch.tensor([1.0, 2.0, 0.5, 4.0])[torch.arange(n) % 4].view(n, 1, 1)
    k = (a.float() * scale).to(a.dtype)
    for row, kind in specials.items():
        k[row] = {"neg": -a[0], "neg2": (-2 * a[0].float()).to(a.dtype), "zero": torch.zeros_like(a[0])}[kind]
    return k.contiguous()


@pytest.mark.parametrize("dtype,d,hq,hkv", [(torch.float32, 64, 2, 1), (torch.float32, 128, 4, 2), (torch.bfloat16, 64, 4, 2),
                                            (torch.bfloat16, 128, 4, 1)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3, 4, 5])
def test_query_agnostic_score_with_keys_parallel_to_the_anchor(dtype, d, hq, hkv, seed):
    # Every ordinary key is a positive multiple of a, so the anchor is parallel to a and 1 - cos rounds to zero or
    # to a few ulps on either side of it; the only dissimilar keys are -a (score 2), the zero key (score 1) and,
    # in the second block, -2a (score 2, younger than -a).  With two places for candidates the retained sets are
    # fixed: {-a, zero} after the first block, {-a, -2a} after the second.  The cut-off gap is about 1, so the
    # oracle's set has to be matched exactly.
    w, B, c = 4, 6, 40
    kvc = Kvc(1, hq, hkv, d, dtype, B, c, w, policy=binding.KVC_SCORE_KEYDIFF)
    orc = KVCOracle(1, hq, hkv, d, B, w, policy="keydiff")
    g = torch.Generator().manual_seed(100 + seed)
    a = torch.randn(1, hkv, d, generator=g).to(dtype)
    k1 = _parallel_keys(a, 40, {7: "neg", 21: "zero"})
    q1 = torch.randn(40, hq, d, generator=g).to(dtype); v1 = torch.randn(40, hkv, d, generator=g).to(dtype)
    compare_chunk(kvc, orc, 0, q1, k1, v1, 0)
    _, _, pos, ln = kvc.cache_view(0)
    for h in range(hkv):
        assert sorted(pos[h, :ln].tolist()) == [7, 21, 36, 37, 38, 39]
    k2 = _parallel_keys(a, 30, {11: "neg2"})
    q2 = torch.randn(30, hq, d, generator=g).to(dtype); v2 = torch.randn(30, hkv, d, generator=g).to(dtype)
    compare_chunk(kvc, orc, 0, q2, k2, v2, 40)
    _, _, pos, ln = kvc.cache_view(0)
    for h in range(hkv):
        assert sorted(pos[h, :ln].tolist()) == [7, 40 + 11, 66, 67, 68, 69]
    # no score may be negative: the selection orders scores by their bit patterns
    _, score = kvc.workspace_view(0)
    assert float(score[:, :32].min()) >= 0.0


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.bfloat16, 128)])
def test_query_agnostic_score_identical_keys_keep_the_oldest(dtype, d):
    # all keys identical: every candidate has exactly the same score, so the older entries stay (the tie rule),
    # whatever sign the rounding of 1 - cos takes
    hq = hkv = 2; w, B, c = 2, 9, 32
    for seed in range(6):
        kvc = Kvc(1, hq, hkv, d, dtype, B, c, w, policy=binding.KVC_SCORE_KEYDIFF)
        g = torch.Generator().manual_seed(300 + seed)
        a = torch.randn(1, hkv, d, generator=g).to(dtype)
        k = a.repeat(32, 1, 1).contiguous()
        q = torch.randn(32, hq, d, generator=g).to(dtype); v = torch.randn(32, hkv, d, generator=g).to(dtype)
        kvc.prefill_chunk(0, q.cuda(), k.cuda(), v.cuda(), 0)
        torch.cuda.synchronize()
        assert kvc.status() == 0
        _, _, pos, ln = kvc.cache_view(0)
        _, score = kvc.workspace_view(0)
        assert ln == B
        for h in range(hkv):
            assert sorted(pos[h, :ln].tolist()) == list(range(B - w)) + [30, 31]
            assert float(score[h, :30].min()) >= 0.0 and float(score[h, :30].max()) <= 1e-5


# ------------------------------------------------------------------------------------------------
# scores that leave the running maximum far behind

@pytest.mark.parametrize("hq,hkv,blocks", [(2, 2, (512, 512)), (8, 2, (256, 200, 256)), (4, 1, (128, 128, 128, 77))])
def test_a_key_whose_score_dwarfs_everything_before_it(hq, hkv, blocks):
    # The attention kernel keeps a reference maximum per row and raises it (rescaling O and the row sum) only when a
    # tile's maximum exceeds it by more than a threshold.  Here every query is the same +-1 vector u, ordinary keys
    # are small, and a few keys are large multiples of u, each larger than the last, placed in the first and in the
    # second half of key tiles that are not a row's first: their scores (5 |u|^2 / sqrt(d) = 57 nats and up) exceed
    # everything before them by far more than any lazy rule may let pass, for the rows that can see them and not for
    # the others of the same warp.  The softmax saturates on those keys; outputs, scores and retained sets must match.
    d, B, w = 128, 1024, 8
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, B, max(blocks), w)
    orc = KVCOracle(1, hq, hkv, d, B, w)
    g = torch.Generator().manual_seed(7)
    u = (torch.randint(0, 2, (d,), generator=g) * 2 - 1).float()
    big = {200: 5.0, 300: 8.0, 470: 12.0, 600: 16.0, 900: 24.0}     # token -> multiple of u (tile halves: 2nd, 1st, 2nd, 2nd, 1st)
    p = 0
    for n in blocks:
        q = u.expand(n, hq, d).clone().bfloat16()
        k = (0.25 * torch.randn(n, hkv, d, generator=g)).bfloat16()
        v = torch.randn(n, hkv, d, generator=g).bfloat16()
        for tok, mult in big.items():
            if p <= tok < p + n:
                k[tok - p] = (mult * u).bfloat16()
        stats = compare_chunk(kvc, orc, 0, q, k, v, p)
        assert kvc.status() == 0
        p += n
    assert stats is not None

# ------------------------------------------------------------------------------------------------
# the bounded wait

def test_a_wait_that_runs_out_reports_timeout_and_leaves_the_context_usable():
    # Every wait in the kernels gives up after the context's limit.  The self-test kernel waits on a barrier that
    # nothing will ever complete, with a limit of about 64k cycles: it must return by itself, the status word must
    # read KVC_ETIMEOUT, and after the status word is cleared an ordinary block must run and match the oracle.
    hq, hkv, d = 4, 2, 128
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, 64, 48, 8)
    install_guards(kvc)
    kvc.set_wait_limit(1 << 16)
    kvc.selftest_wait_timeout()
    torch.cuda.synchronize()
    assert kvc.status() == KVC_ETIMEOUT
    assert "status word" in kvc.last_error()
    check_guards(kvc)
    kvc.workspace_init()
    assert kvc.status() == 0
    kvc.set_wait_limit(2_000_000_000)
    orc = KVCOracle(1, hq, hkv, d, 64, 8)
    torch.manual_seed(5)
    p = 0
    for n in (48, 40):
        q = torch.randn(n, hq, d).bfloat16(); k = torch.randn(n, hkv, d).bfloat16(); v = torch.randn(n, hkv, d).bfloat16()
        compare_chunk(kvc, orc, 0, q, k, v, p)
        p += n
    with pytest.raises(binding.KvcError):
        kvc.set_wait_limit(10)                       # below the accepted range


# ------------------------------------------------------------------------------------------------
# the guard regions themselves

def test_guard_check_notices_a_stray_byte():
    # the checker must fail when a byte outside a buffer changes (here: written by the test itself, on the host side
    # of the comparison, never by a kernel)
    kvc = Kvc(2, 2, 1, 64, torch.float32, 32, 16, 4)
    install_guards(kvc)
    check_guards(kvc)
    whole, view = guarded_copy(torch.zeros(5, 2, 64), kvc.device)
    check_guards(kvc, [(whole, view)])
    kvc._guards["cache"][kvc._guards["stride"] + 3] = 0          # inside the gap after blob 0
    with pytest.raises(AssertionError):
        check_guards(kvc)
    kvc._guards["cache"][kvc._guards["stride"] + 3] = 0xA5
    whole[-1] = 1
    with pytest.raises(AssertionError):
        check_guards(kvc, [(whole, view)])


# ------------------------------------------------------------------------------------------------
# device-side time stamps

@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_device_time_stamps_count_every_launch(dtype):
    # every kernel of the stamped calls leaves a record with begin <= end; the records' durations, added per kind,
    # fit inside the span from the first begin to the last end (the kernels run in stream order), and the results
    # are those of an unstamped run
    hq, hkv, d = 8, 2, 128
    a = Kvc(1, hq, hkv, d, dtype, 256, 160, 16)
    b = Kvc(1, hq, hkv, d, dtype, 256, 160, 16)
    torch.manual_seed(11)
    blocks = [(torch.randn(n, hq, d, device="cuda").to(dtype), torch.randn(n, hkv, d, device="cuda").to(dtype),
               torch.randn(n, hkv, d, device="cuda").to(dtype)) for n in (160, 150, 160, 33)]
    before = b.launch_count()
    b.profile_device(64)
    p = 0
    for q, k, v in blocks:
        oa = a.prefill_chunk(0, q, k, v, p); ob = b.prefill_chunk(0, q, k, v, p)
        assert torch.equal(oa, ob)
        p += q.shape[0]
    ms, cnt, span = b.profile_device_read()
    b.profile_device(0)
    assert sum(cnt.values()) == b.launch_count() - before
    assert cnt["attention"] == 4 and cnt["compress"] == 3
    assert all(ms[s] > 0 for s in cnt if cnt[s]) and sum(ms.values()) <= span * 1.001
    assert torch.equal(a.cache_view(0)[2], b.cache_view(0)[2])
    # off again: the next call must not touch the (freed) record buffer
    q, k, v = blocks[0]
    b.prefill_chunk(0, q, k, v, p)
    torch.cuda.synchronize()
    assert b.status() == 0


@pytest.mark.parametrize("flags", [8, 16])
def test_device_time_stamps_in_plain_order_cover_the_whole_kernel(flags):
    # the query-agnostic score reads all keys twice in front of the kernel's dependency wait: inside the record in plain
    # stream order and on the side stream, outside it where the launch overlaps the attention
    hq, hkv, d, B, n = 8, 4, 128, 3000, 24
    torch.manual_seed(1)
    q, k, v = (torch.randn(B + n, h, d, device="cuda", dtype=torch.bfloat16) for h in (hq, hkv, hkv))
    us = {}
    for fl in (0, flags):
        kvc = Kvc(1, hq, hkv, d, torch.bfloat16, B, n, 32, flags=fl, policy=binding.KVC_SCORE_KEYDIFF)
        kvc.prefill_chunk(0, q[:B], k[:B], v[:B], 0)
        kvc.profile_device(16)
        for i in range(6):
            kvc.prefill_chunk(0, q[B:], k[B:], v[B:], B + i * n)
        kvc.join()
        ms, cnt, _ = kvc.profile_device_read()
        assert cnt["compress"] == 6 and kvc.status() == 0
        us[fl] = 1e3 * ms["compress"] / 6
    assert us[flags] > 1.3 * us[0], us


# ------------------------------------------------------------------------------------------------
# host buffers: blocks of different sizes back to back

def test_host_blocks_of_different_sizes_do_not_overwrite_each_other():
    # a small block's result must not share staging memory with the inputs of the larger block two calls later: its copy
    # to the host may still be on its way when those arrive
    hq, hkv, d, layers, blocks = 12, 4, 128, 6, (300, 4, 300, 30, 300)
    torch.manual_seed(3)
    a, b = (Kvc(layers, hq, hkv, d, torch.bfloat16, 64, max(blocks)) for _ in range(2))
    calls, pos = [], 0
    for n in blocks:
        for layer in range(layers):
            calls.append((layer, pos, [torch.randn(n, h, d).to(torch.bfloat16).pin_memory() for h in (hq, hkv, hkv)]))
        pos += n
    want = [a.prefill_chunk(layer, *(t.cuda() for t in qkv), p) for layer, p, qkv in calls]
    outs = [torch.empty_like(qkv[0]).pin_memory() for _, _, qkv in calls]
    for _ in range(20):
        for o in outs:
            o.zero_()
        b.reset()
        for (layer, p, qkv), o in zip(calls, outs):
            b.prefill_chunk_host(layer, *qkv, p, o)
        b.host_flush()
        torch.cuda.synchronize()
        assert b.status() == 0
        for (layer, p, _), o, w in zip(calls, outs, want):
            assert torch.equal(o, w.cpu()), f"layer {layer}, position {p}"


def test_a_rejected_host_call_does_not_expose_the_result_of_the_call_before_it():
    # the call after a rejected one must not put its result where that of the last accepted call may still be on its way to
    # the host: both results lie in the staging buffer afterwards
    hq, hkv, d, n = 8, 2, 64, 40
    torch.manual_seed(4)
    a, b = (Kvc(1, hq, hkv, d, torch.bfloat16, 64, n) for _ in range(2))
    blocks = [[torch.randn(n, h, d).to(torch.bfloat16).pin_memory() for h in (hq, hkv, hkv)] for _ in range(2)]
    want = [a.prefill_chunk(0, *(t.cuda() for t in qkv), i * n).cpu() for i, qkv in enumerate(blocks)]
    outs = [torch.empty_like(qkv[0]).pin_memory() for qkv in blocks]
    b.prefill_chunk_host(0, *blocks[0], 0, outs[0])
    with pytest.raises(binding.KvcError):
        b.prefill_chunk_host(0, *blocks[1], -1, outs[1])
    b.prefill_chunk_host(0, *blocks[1], n, outs[1])
    b.host_flush()
    torch.cuda.synchronize()
    assert b.status() == 0 and all(torch.equal(o, w) for o, w in zip(outs, want))
    staged = b.staging.cpu().numpy().tobytes()
    assert all(w.view(torch.uint8).numpy().tobytes() in staged for w in want)


# ------------------------------------------------------------------------------------------------
# inputs reused in stream order right behind a call

@pytest.mark.parametrize("dtype,policy,flags", [(torch.bfloat16, 0, 0), (torch.bfloat16, 0, 16), (torch.bfloat16, 1, 0),
                                                 (torch.bfloat16, 1, 16), (torch.float32, 0, 0), (torch.float32, 1, 0)])
def test_inputs_may_be_reused_behind_a_call(dtype, policy, flags):
    # k and v (and q, unless compress runs on a side stream) may be overwritten by the stream's next work although the
    # scoring reads q and k: results equal those of calls whose inputs stay
    hq, hkv, d, n, B, layers = 8, 4, 128, 200, 300, 2
    torch.manual_seed(5)
    data = [[torch.randn(n, h, d, device="cuda").to(dtype) for h in (hq, hkv, hkv)] for _ in range(5 * layers)]
    res = []
    for reuse in (False, True):
        kvc = Kvc(layers, hq, hkv, d, dtype, B, n, policy=policy, flags=flags)
        buf = [[torch.empty_like(t) for t in data[0]] for _ in range(layers)]
        outs, kept = [], []
        for i, qkv in enumerate(data):
            layer = i % layers
            ins = buf[layer] if reuse else [t.clone() for t in qkv]
            kept.append(ins)                    # (the allocator must not hand a clone's memory on before the side stream is done)
            if reuse:
                for b, t in zip(ins, qkv):
                    b.copy_(t)
            out = kvc.prefill_chunk(layer, *ins, (i // layers) * n)
            if reuse:
                for t in (ins[1:] if flags & 16 else ins):
                    t.fill_(7.0)
                if flags & 16:
                    kvc.join()                  # q is overwritten by the next use of the buffer
            outs.append(out)
        kvc.join()
        assert kvc.status() == 0
        res.append((outs, [kvc.cache_view(l)[2][:, :B].clone() for l in range(layers)]))
    assert all(torch.equal(a, b) for a, b in zip(res[0][0], res[1][0]))
    assert all(torch.equal(a, b) for a, b in zip(res[0][1], res[1][1]))


# ------------------------------------------------------------------------------------------------
# workspace slots while a compress kernel is pending on a side stream

def _longest_chain(graph):
    """Nodes on the longest path of a captured graph."""
    rt, handle, n = ctypes.CDLL("libcudart.so.12"), ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert rt.cudaGraphGetEdges(handle, None, None, ctypes.byref(n)) == 0
    src, dst = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetEdges(handle, src, dst, ctypes.byref(n)) == 0
    after = {}
    for a, b in zip(src, dst):
        after.setdefault(a, []).append(b)

    def depth(node):
        return 1 + max((depth(x) for x in after.get(node, ())), default=0)

    return max(depth(node) for node in after)


@pytest.mark.parametrize("single,batched,chain", [(0, 2, 4), (1, 2, 4), (3, 0, 3)])
def test_a_batched_call_waits_for_the_workspace_slots_it_uses(single, batched, chain):
    # a batched call works in the first slots: behind the compress kernel of a layer that has one of them as its own, beside
    # that of any other.  The calls are captured and never run: attention, compress, attention, compress in one chain or two
    n, B = 64, 128
    kvc = Kvc(4, 4, 2, 64, torch.bfloat16, B, n, flags=KVC_FLAG_ASYNC_COMPRESS | 8)      # 8: plain edges
    q, k, v = (torch.randn(2, n, h, 64, device="cuda", dtype=torch.bfloat16) for h in (4, 2, 2))
    out = torch.empty_like(q)
    for p in (0, n, 2 * n):                                       # every layer evicts from here on; kernels are loaded
        for l in range(4):
            kvc.prefill_chunk(l, q[0], k[0], v[0], p)
    kvc.prefill_chunk_layers(0, q, k, v, 3 * n, out)
    kvc.prefill_chunk_layers(2, q, k, v, 3 * n, out)
    assert kvc.status() == 0
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        kvc.prefill_chunk(single, q[0], k[0], v[0], 4 * n, out[0])
        kvc.prefill_chunk_layers(batched, q, k, v, 4 * n, out)
        kvc.join()
    assert _longest_chain(graph) == chain


def test_a_compress_left_pending_before_a_capture():
    # a captured batched call cannot wait for work from outside the capture: the host has waited for it when the call returns
    n, B = 64, 128
    a, b = (Kvc(4, 4, 2, 64, torch.bfloat16, B, n, flags=KVC_FLAG_ASYNC_COMPRESS) for _ in range(2))
    torch.manual_seed(3)
    q, k, v = (torch.randn(2, n, h, 64, device="cuda", dtype=torch.bfloat16) for h in (4, 2, 2))
    out = [torch.empty_like(q) for _ in range(2)]
    for kvc, o in ((a, out[0]), (b, out[1])):
        for p in (0, n, 2 * n):
            for l in range(4):
                kvc.prefill_chunk(l, q[0], k[0], v[0], p)
        kvc.join()
        kvc.prefill_chunk(0, q[0], k[0], v[0], 3 * n)                # left pending
        if kvc is a:
            kvc.prefill_chunk_layers(2, q, k, v, 3 * n, o)
            continue
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            kvc.prefill_chunk_layers(2, q, k, v, 3 * n, o)
            kvc.join()
        graph.replay()
    assert a.status() == 0 and b.status() == 0
    assert torch.equal(*out)
    for l in (0, 2, 3):
        assert all(torch.equal(x[:, :B], y[:, :B]) for x, y in zip(a.cache_view(l)[:3], b.cache_view(l)[:3]))


def test_batched_and_host_calls_beside_a_pending_compress():
    # the same calls on a context without the flag give the same bits
    layers, hq, hkv, d, B, n = 4, 8, 8, 64, 3000, 200
    N = B + 6 * n
    torch.manual_seed(11)
    Q, K, V = (torch.randn(layers, N, h, d, device="cuda", dtype=torch.bfloat16) for h in (hq, hkv, hkv))
    host = [x[1].cpu().pin_memory() for x in (Q, K, V)]
    held = []
    for flags in (0, KVC_FLAG_ASYNC_COMPRESS):
        kvc = Kvc(layers, hq, hkv, d, torch.bfloat16, B, n, flags=flags)
        out, out_host = torch.zeros_like(Q), torch.zeros_like(host[0]).pin_memory()
        for l in range(layers):                                   # the cache is full, nothing evicted yet
            kvc.prefill_chunk(l, Q[l, :B], K[l, :B], V[l, :B], 0, out[l, :B])
        for i, p in enumerate(range(B, N, n)):
            s = slice(p, p + n)
            kvc.prefill_chunk(0, Q[0, s], K[0, s], V[0, s], p, out[0, s])
            if i % 2:
                kvc.prefill_chunk_host(1, *(x[s] for x in host), p, out_host[s])
            kvc.prefill_chunk_layers(2, Q[2:, s], K[2:, s], V[2:, s], p, out[2:, s])
            if i % 2 == 0:
                kvc.prefill_chunk_host(1, *(x[s] for x in host), p, out_host[s])
        kvc.host_flush()
        assert kvc.status() == 0
        held.append([out, out_host] + [t[:, :B] for l in range(layers) for t in kvc.cache_view(l)[:3]])
    assert all(torch.equal(a, b) for a, b in zip(*held))
