"""How the kernels leave when a bounded wait has run out.  Nothing of theirs may still be under way when they give up what
it uses: tensor memory under MMAs, shared memory under copies.  That cannot be provoked on a GPU, so the kernels' own sources
run here on the host, one CTA with a thread per CUDA thread (cta_emulator/emu.h), with late copies and slow MMAs."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2604_16734_b200", "csrc")
CUDA = "/usr/local/cuda/include"
KVC_ETIMEOUT = -4


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "cuda_bf16.h")):
        pytest.skip("needs g++ and the CUDA headers")
    tmp = tmp_path_factory.mktemp("emulator")

    def source(name):
        text = open(os.path.join(CSRC, name)).read()
        text = re.sub(r"^#(include|pragma once).*$", "", text, flags=re.M)
        text = re.sub(r"asm volatile\(\"mov\.u64 %0, %%globaltimer.*$", "t = 0;", text, flags=re.M)
        return text.replace("extern __shared__ uint8_t smem_raw[];", "extern uint8_t* smem_raw;")

    # the bounded waits are the library's, on the emulator's barriers
    ptx = source("ptx.cuh")
    waits = re.findall(r"^__device__ __forceinline__ (?:bool|void) (?:mbar_wait|mbar_wait_spin|word_wait_spin|mbar_drain)\(.*?^}\n", ptx, flags=re.M | re.S)
    limit = re.search(r"^static constexpr int kDefaultWaitLimitK.*$", ptx, flags=re.M).group(0)
    parts = ["namespace kvc {", limit, *waits, "}", source("geom.cuh"), source("kernels_tc.cuh"), source("compress.cuh")]
    (tmp / "kernels.h").write_text("\n".join(parts))
    exe = str(tmp / "emulator")
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-I", str(tmp), "-I", CUDA, "-I", os.path.join(HERE, "cta_emulator"),
                    os.path.join(HERE, "cta_emulator", "main.cpp"), "-o", exe], check=True)

    def run(**kw):
        r = subprocess.run(["timeout", "20", exe] + [f"{k}={v}" for k, v in kw.items()], capture_output=True, text=True)
        assert r.returncode != 124, "the kernel does not end"
        lines = r.stdout.splitlines()
        assert lines and lines[-1].startswith("status"), r.stdout + r.stderr
        return [x[len("FAULT "):] for x in lines[:-1]], int(lines[-1].split()[1])
    return run


SHAPES = [dict(row_tiles=1, n=128, n_c=300), dict(row_tiles=2, n=256, n_c=300), dict(row_tiles=1, n=128, n_c=900, split=2)]


@pytest.mark.parametrize("shape", SHAPES)
def test_attention_that_nothing_holds_up(emulator, shape):
    assert emulator(kernel="attention", limit_ms=5000, **shape) == ([], 0)


@pytest.mark.parametrize("shape", SHAPES)
def test_attention_keeps_tensor_memory_until_its_mmas_are_done(emulator, shape):
    # the first K tile lands after the softmax warps have given up, while the issuer of S is still suspended on it
    issuers = ",".join(f"{w}:400" for w in (9, 10))
    faults, status = emulator(kernel="attention", limit_ms=20, load_ms="0:60,1:60", suspend_ms=issuers, **shape)
    assert status == KVC_ETIMEOUT and not [f for f in faults if "TMEM" in f]
    # MMAs that outlast the limit
    faults, status = emulator(kernel="attention", limit_ms=20, mma_us=40000, **shape)
    assert status == KVC_ETIMEOUT and not [f for f in faults if "TMEM" in f or "MMA" in f]


@pytest.mark.parametrize("shape", SHAPES)
def test_attention_waits_for_its_loads(emulator, shape):
    # loads that land long after everybody has given up: Q and the first tiles, or the last key tile's
    key_tiles = ((shape["n"] + 127) // 128 + (shape["n_c"] + 127) // 128) // shape.get("split", 1)
    loads = shape["row_tiles"] + 2 * key_tiles
    for late in ((0, 1, 2, 3), (loads - 2, loads - 1)):
        faults, status = emulator(kernel="attention", limit_ms=20, load_ms=",".join(f"{i}:150" for i in late), **shape)
        assert (faults, status) == ([], KVC_ETIMEOUT), late


def test_attention_waits_for_the_copies_of_its_cluster(emulator):
    # its own key tiles are late, so that it has given up when the other CTAs' partial rows are still on their way to it
    faults, status = emulator(kernel="attention", limit_ms=20, load_ms="1:60", copy_ms=200, **SHAPES[2])
    assert (faults, status) == ([], KVC_ETIMEOUT)
    # nothing but those copies is late
    faults, status = emulator(kernel="attention", limit_ms=30, copy_ms=200, **SHAPES[2])
    assert (faults, status) == ([], KVC_ETIMEOUT)


def test_compress_that_nothing_holds_up(emulator):
    assert emulator(kernel="compress", limit_ms=5000, n_c=900, budget=900) == ([], 0)


@pytest.mark.parametrize("late", [dict(load_ms="0:150,1:150,2:150"), dict(load_ms="3:150,4:150"), dict(mma_us=40000)])
def test_compress_waits_for_its_loads_and_mmas(emulator, late):
    # the selection lays its tables over the tiles, and tensor memory goes back before it
    faults, status = emulator(kernel="compress", limit_ms=20, n_c=900, budget=900, **late)
    assert (faults, status) == ([], KVC_ETIMEOUT)


def test_score_that_nothing_holds_up(emulator):
    assert emulator(kernel="score", limit_ms=5000, n=512, w=512) == ([], 0)


@pytest.mark.parametrize("late", [dict(load_ms="0:150,1:150"), dict(load_ms="2:150"), dict(mma_us=40000),
                                  dict(mma_us=20000, suspend_ms="3:400")])
def test_score_waits_for_its_loads_and_mmas(emulator, late):
    # (the last one: a warp still sees the first group's products, and those that have given up leave with it)
    faults, status = emulator(kernel="score", limit_ms=20, n=512, w=512, **late)
    assert (faults, status) == ([], KVC_ETIMEOUT)
