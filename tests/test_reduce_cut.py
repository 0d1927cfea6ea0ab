"""The cut of a reduce over CTAs and threads (csrc/reduce_cut.h), compiled for the host:
every index of a window belongs to one thread, the grid is one wave at most, and a
window of few Gray blocks is dealt to enough lanes."""

import ctypes
import random
import subprocess

import pytest

from paper_2103_00693_gb300 import build as hbuild

SHIM = """
#include <chrono>
#include "reduce_cut.h"
using Clock = std::chrono::steady_clock;
extern "C" double divisions(uint64_t chunk, uint64_t n, int U, uint64_t T, uint64_t sms, uint64_t room, uint64_t smem)
{
    volatile uint64_t c = chunk, by = 3, sink = 0;
    double best = 1e30;
    for (int rep = 0; rep < 20; ++rep) {
        uint64_t x = 0, y = ~0ull;
        const auto t0 = Clock::now();
        for (int i = 0; i < 500; ++i) x += hlf::reduce_shape(c, n, U, T, sms, room, smem).per;
        const auto t1 = Clock::now();
        for (int i = 0; i < 500 * 100; ++i) y = (y + ~0ull) / by;
        const auto t2 = Clock::now();
        sink = x + y;
        const double r = 100.0 * (t1 - t0).count() / (t2 - t1).count();
        if (r < best) best = r;
    }
    return best;
}
extern "C" void cut(uint64_t chunk, uint64_t n, int U, uint64_t T, uint64_t sms, uint64_t room, uint64_t smem, uint64_t* o)
{
    const hlf::ReduceShape s = hlf::reduce_shape(chunk, n, U, T, sms, room, smem);
    o[0] = s.threads; o[1] = s.blocks; o[2] = s.parts; o[3] = s.per; o[4] = s.runs; o[5] = s.align;
}
"""
SMS = 152
SHAPES = [(1, 3, 1024, 1024), (1, 6, 1024, 1024), (2, 4, 1024, 1024), (4, 3, 1024, 1024), (5, 2, 256, 512), (11, 2, 256, 512), (16, 2, 256, 512)]


def _smem(shape):
    """A CTA's tables and partial results in bytes."""
    W, _, T, _ = shape
    return 66 * W * 8 + 16 * 16 * W * 8 + T // 32 * (2 + W) * 8


def _fit(shape, threads):
    """CTAs that an SM of 228 KB, 1 KB of it for each CTA, holds at once."""
    return min(shape[3] // threads, 228 * 1024 // (_smem(shape) + 1024))


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("cut")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", hbuild.CSRC, str(d / "shim.cpp"), "-o",
                    str(d / "cut.so")], check=True)
    lib = ctypes.CDLL(str(d / "cut.so"))

    lib.divisions.restype = ctypes.c_double

    def f(chunk, n, shape, divisions=False):
        W, U, T, room = shape
        o = (ctypes.c_uint64 * 6)()
        u64 = ctypes.c_uint64
        if divisions:
            return lib.divisions(u64(chunk), u64(n), U, u64(T), u64(SMS), u64(room), u64(_smem(shape)))
        lib.cut(u64(chunk), u64(n), U, u64(T), u64(SMS), u64(room), u64(_smem(shape)), o)
        return dict(zip(("threads", "blocks", "parts", "per", "runs", "align"), o))

    return f


def _runs(s, first, chunk):
    """The kernel's own arithmetic: (first index, length) of each thread's run."""
    skip = first & s["align"]
    for run in range(s["parts"] * s["threads"]):
        a = run * s["per"]
        lo = max(a, skip)
        if run < s["runs"] and lo - skip < chunk:
            yield first + lo - skip, min(s["per"] - (lo - a), chunk - (lo - skip))


@pytest.mark.parametrize("shape", SHAPES)
def test_every_index_once(cut, shape):
    rng = random.Random(shape[0])
    sizes = [1, 2, 3, 4, 7, 8, 15, 16, 31, 32, 33, 63, 64, 96, 97, 224, 225, 255, 256, 480, 481, 768, 769, 1023, 3840, 3841, 8191]
    for chunk in sizes + [int(2 ** rng.uniform(0, 34)) for _ in range(12)]:
        for n in (1, 7, 153, 100000):
            s = cut(chunk, n, shape)
            assert 32 <= s["threads"] <= shape[2] and s["threads"] % 32 == 0
            assert 1 <= s["blocks"] <= min(n * s["parts"], SMS * _fit(shape, s["threads"]))
            first = rng.randrange(1 << 40)
            at = first
            for i, length in _runs(s, first, chunk):
                assert i == at and length >= 1, (chunk, n, s)
                at += length
            assert at == first + chunk, (chunk, n, s)


@pytest.mark.parametrize("shape", SHAPES)
def test_short_windows_fill_lanes(cut, shape):
    """A thread of a short window walks no more than a warp's share of it; where all
    windows run at once, no more than a CTA's."""
    U = shape[1]
    for chunk in (2, 10, 31, 32 * ((1 << U) - 1)):
        assert cut(chunk, 100000, shape)["per"] <= (chunk + 31) // 32
    for chunk in (2, 10, 100, 256 * (((1 << U) + 2) // 3)):
        assert cut(chunk, 7, shape)["per"] <= (chunk + 255) // 256


@pytest.mark.parametrize("shape", SHAPES)
def test_cta_no_larger_than_its_window(cut, shape):
    """Windows that all run at once: 256 threads, or one for each Gray block; lanes walk
    whole blocks where they would have more than a third of a block each."""
    U = shape[1]
    for chunk in (300, 2000):
        for n in (7, 100, 400):
            s = cut(chunk, n, shape)
            if s["parts"] > 1 or n > SMS * _fit(shape, s["threads"]):
                continue
            assert s["threads"] <= max(256, ((chunk - 1 >> U) + 2 + 31) // 32 * 32)
            assert s["align"] or s["per"] <= ((1 << U) + 2) // 3


@pytest.mark.parametrize("shape", SHAPES)
def test_one_window_has_threads_for_its_tables(cut, shape):
    for chunk in (1, 4, 20):
        s = cut(chunk, 1, shape)
        assert s["threads"] >= 256 and s["parts"] == 1


def _every_cut(chunk, n, shape):
    """(threads, parts) of the first cheapest cut, each tried by itself."""
    W, U, T, _ = shape
    runs, best, pick = ((chunk - 1) >> U) + 2, 1 << 64, None
    bd = T
    while bd >= 64:
        slots, least, k = SMS * _fit(shape, bd), best - best // 16, 1
        while k <= 64 and (k == 1 or (k - 1) * bd < runs):
            cost = -(-n * k // slots) * (48 + ((chunk - 1) // (k * bd) | (1 << U) - 1) + 1)
            if cost < best and (bd == T or cost < least):
                best, pick = cost, (bd, k)
            k += 1
        bd //= 2
    return pick


@pytest.mark.parametrize("shape", SHAPES)
def test_the_cheapest_of_all_cuts(cut, shape):
    rng = random.Random(77)
    for _ in range(150):
        n, chunk = int(2 ** rng.uniform(1, 17)), int(2 ** rng.uniform(13, 34))
        s = cut(chunk, n, shape)
        threads, parts = _every_cut(chunk, n, shape)
        assert s["parts"] == parts, (chunk, n)
        if parts > 1 or n > SMS * _fit(shape, threads):  # else the CTA may be smaller than the cut's
            assert s["threads"] == threads, (chunk, n)


@pytest.mark.parametrize("chunk,n,shape", [(100000, 153, SHAPES[0]), (1 << 20, 7, SHAPES[2]), (77474, 64, SHAPES[-1])])
def test_host_time(cut, chunk, n, shape):
    """Short reduces: the cut costs the host less than 120 divisions (each cut tried by
    itself took 220 to 540, this takes 20 to 40)."""
    assert cut(chunk, n, shape, divisions=True) < 120
