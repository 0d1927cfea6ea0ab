"""The histogram's sum over aligned blocks: one block, windows of many block
sizes, fields whose span never fills (bits that no row changes), the narrowest and
widest fields, and windows far larger than could be counted one by one, which
must equal the sum of their parts."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
import synth
from oracle import cpu as oc

pytestmark = pytest.mark.gpu


def _sparse(n, r):
    """Rank r: a path on the first vertices, the rest isolated and zero."""
    A = np.zeros((n, n), dtype=np.uint8)
    A[np.arange(r), np.arange(r)] = 1
    return A


@pytest.mark.parametrize("order", [hlf.ORDER_GRAY, hlf.ORDER_PAPER])
@pytest.mark.parametrize("A,fields", [
    (synth.grid_instance(8, 0.5, 0), [(0, 1), (63, 1), (0, 20), (44, 20), (13, 7)]),
    (_sparse(40, 18), [(0, 20), (10, 16), (17, 2), (20, 20)]),
    (synth.random_symmetric(130, 0.5, 3), [(120, 10), (55, 18), (64, 20)]),
], ids=["grid8", "sparse40", "sym130"])
def test_blocks(cuda_ok, A, fields, order):
    F = oc.factor(A)
    G = hlf.Factorization.from_dense(A)
    G.set_order(order)
    space = 1 << F.space_log2()
    for off, cnt in ((0, 1), (space - 1, 1), (1, 1), (0, 4096), (4095, 2), (77, 65536 - 154), (space // 2 - 3333, 9999)):
        for lo, nb in fields:
            got = G.histogram(off, cnt, lo, nb).cpu().numpy().view(np.uint64)
            want = oc.histogram(F, off, cnt, lo, nb, "paper" if order == hlf.ORDER_PAPER else "gray")
            assert np.array_equal(got, want), (off, cnt, lo, nb)
    G.close()


def test_large_windows_add_up(cuda_ok):
    A = synth.grid_instance(9, 0.5, 2)
    F = oc.factor(A)
    assert F.r >= 60
    G = hlf.Factorization.from_dense(A)
    cut = [5, 70001, 70001 + (1 << 33), (1 << 50) + 12345, (1 << 59) + 1]
    for lo, nb in ((0, 14), (60, 12), (33, 16)):
        whole = G.histogram(cut[0], cut[-1] - cut[0], lo, nb).cpu().numpy().view(np.uint64)
        parts = [G.histogram(a, b - a, lo, nb).cpu().numpy().view(np.uint64) for a, b in zip(cut, cut[1:])]
        assert np.array_equal(parts[0], oc.histogram(F, cut[0], cut[1] - cut[0], lo, nb))
        assert np.array_equal(whole, sum(parts[1:], parts[0])) and int(whole.sum()) == cut[-1] - cut[0]
    G.close()
