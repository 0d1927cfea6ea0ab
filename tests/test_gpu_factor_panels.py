"""Stage 1 where the panel search can go wrong: sizes around the panel, warp and word
edges, matrices whose first searched rows do not span a panel (few distinct rows,
low rank, pivots that only the last rows have), columns without pivots, and faulty
input (bits past n, one asymmetric bit), which must end with its status."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
from oracle import cpu as oc

pytestmark = pytest.mark.gpu


def _sym(U):
    U = np.triu(U.astype(np.uint8))
    return U | U.T


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "ones":
        return np.ones((n, n), dtype=np.uint8)
    if kind == "few":  # rank <= 7, every row one of 128 combinations
        B = rng.integers(0, 2, (7, n))
        C = _sym(rng.integers(0, 2, (7, 7)))
        return ((B.T @ C @ B) % 2).astype(np.uint8)
    if kind == "half":  # rank about n / 2
        B = rng.integers(0, 2, (n // 2 + 1, n))
        C = _sym(rng.integers(0, 2, (n // 2 + 1, n // 2 + 1)))
        return ((B.T @ C @ B) % 2).astype(np.uint8)
    if kind == "anti":  # the pivot of column c is row n - 1 - c only
        return np.eye(n, dtype=np.uint8)[::-1].copy()
    if kind == "late":  # equal rows, and the rest of the rank in the last few rows
        A = np.ones((n, n), dtype=np.uint8)
        k = max(1, n // 10)
        S = _sym(rng.integers(0, 2, (n, n)))
        A[-k:, :] = S[-k:, :]
        A[:, -k:] = S[-k:, :].T
        return A
    return _sym(rng.integers(0, 2, (n, n)))


def _check(A):
    F = oc.factor(A)
    G = hlf.Factorization.from_dense(A)
    assert G.rank == F.r
    piv, z0, basis = G.factor_host()
    assert np.array_equal(piv, F.piv) and np.array_equal(z0, F.z0_words()) and np.array_equal(basis, F.basis_words())
    if F.r:
        G.set_order(hlf.ORDER_PAPER)
        k = min(1 << F.space_log2(), 300)
        off = (1 << F.space_log2()) - k
        assert np.array_equal(G.store(off, k).cpu().numpy().view(np.uint64), oc.paper_order(F, off, k))
    G.close()


@pytest.mark.parametrize("kind", ["ones", "few", "half", "anti", "late", "dense"])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 129, 160, 191, 193, 256, 257, 289, 384, 512, 513, 641, 1024])
def test_panels(cuda_ok, kind, n):
    _check(_matrix(kind, n))


@pytest.mark.parametrize("n", [40, 100, 250, 300, 700, 1000])
def test_faulty_input(cuda_ok, n):
    import torch

    A = _matrix("dense", n)
    for fault, status in (("padding", "HLF_ERR_PADDING"), ("asymmetric", "HLF_ERR_NOT_SYMMETRIC")):
        words = hlf.pack_rows(A)
        if fault == "padding":
            words[:, -1] |= np.uint64(0xFFFFFFFFFFFFFFFF) << np.uint64(n % 64)
        else:
            words[n - 1, 0] ^= np.uint64(1)
        G = hlf.Factorization(torch.from_numpy(words.view(np.int64)).cuda(), n)
        with pytest.raises(hlf.HlfError) as e:
            G.rank
        assert e.value.status == hlf.hlf.STATUS_CODES[status]
        G.close()
    _check(A)
