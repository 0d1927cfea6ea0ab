"""The cut of a reduce over threads and CTAs: windows around one Gray block, one
CTA's worth of blocks, one wave, the change of unroll, and chunk counts that give a
window one CTA, several, or less than one; element by element against the oracle."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
import synth
from oracle import cpu as oc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def made(cuda_ok):
    out = {}
    for n in (40, 100, 250, 300, 1000):
        A = synth.random_symmetric(n, 0.1, n)
        out[n] = (oc.factor(A), hlf.Factorization.from_dense(A))
    yield out
    for _, G in out.values():
        G.close()


def _check(F, red, off, cnt):
    got = hlf.ReduceResult.from_words(red, F.W)
    c, h, f = oc.reduce(F, off, cnt)
    assert (got.count, got.hsum) == (c, h), (F.n, off, cnt)
    assert np.array_equal(got.xor_fold, f), (F.n, off, cnt)
    assert not np.asarray(red)[2 + F.W:].any()


@pytest.mark.parametrize("n", [40, 100, 250, 300, 1000])
def test_one_window(made, n):
    F, G = made[n]
    T = 1024 if F.W <= 4 else 256
    edges = [1, 3, 4, 7, 8, 9, 8 * T - 8, 8 * T - 7, 8 * T + 1, 4 * T + 1, 16 * T + 5, 152 * T + 3]
    if F.W <= 2:
        edges.append(152 * 8 * T + 11)
    for cnt in edges:
        for off in (0, 5, 8, (1 << F.space_log2()) - cnt):
            _check(F, G.reduce(off, cnt).cpu().numpy(), off, cnt)


def test_unroll_change(made):
    F, G = made[40]
    wave = 152 * 1024
    for cnt in (wave * 1024 - 1, wave * 1024 + 1):
        _check(F, G.reduce(77, cnt).cpu().numpy(), 77, cnt)


@pytest.mark.parametrize("n", [40, 250, 1000])
@pytest.mark.parametrize("chunk,n_chunks", [(1, 3000), (2, 153), (9, 1), (63, 40), (8193, 3), (50001, 153), (70000, 7),
                                           (10, 5000), (96, 2000), (97, 2000), (300, 400), (512, 9), (513, 9), (769, 9), (2001, 100)])
def test_chunks(made, n, chunk, n_chunks):
    F, G = made[n]
    off = 3
    red = G.reduce_chunks(off, chunk, n_chunks).cpu().numpy()
    for c in sorted({0, 1, n_chunks // 2, n_chunks - 1} & set(range(n_chunks))):
        _check(F, red[c], off + c * chunk, chunk)
    assert red[:, 0].tolist() == [chunk] * n_chunks
    total = G.reduce(off, chunk * n_chunks).cpu().numpy().view(np.uint64)
    with np.errstate(over="ignore"):
        assert int(red.view(np.uint64)[:, 1].sum(dtype=np.uint64)) == int(total[1])
    assert np.array_equal(np.bitwise_xor.reduce(red.view(np.uint64)[:, 2:], axis=0), total[2:])
