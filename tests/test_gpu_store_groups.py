"""Where the cut of a stored window into groups can go wrong: windows of less than a
group, exactly one, one more, of both parities of offset and of output address,
at the end of the index space and of 2^64, for one and several words, alone and
many in one launch."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
import synth
from oracle import cpu as oc

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 63, 64, 65, 66, 127, 128, 129, 2047, 2050, 4161, 70001]


@pytest.fixture(scope="module")
def made(cuda_ok):
    out = {}
    for n in (20, 64, 100, 300, 1024):
        A = synth.random_symmetric(n, 0.1, n + 1)
        out[n] = (oc.factor(A), hlf.Factorization.from_dense(A))
    yield out
    for _, G in out.values():
        G.close()


def _offsets(F, cnt):
    space = 1 << F.space_log2()
    return sorted({o for o in (0, 1, 2, 63, 64, 65, 1000, space - cnt, space - cnt - 1) if 0 <= o <= space - cnt})


@pytest.mark.parametrize("n", [20, 64, 100, 300, 1024])
def test_one_window(made, n):
    import torch

    F, G = made[n]
    for cnt in SIZES:
        for off in _offsets(F, cnt):
            buf = torch.full((cnt + 2, F.W), -1, dtype=torch.int64, device="cuda")
            G.store(off, cnt, buf)
            got = buf.cpu().numpy().view(np.uint64)
            assert np.array_equal(got[:cnt], oc.window(F, off, cnt)), (off, cnt)
            assert np.all(got[cnt:] == np.uint64(0xFFFFFFFFFFFFFFFF)), (off, cnt)


def test_output_on_eight_bytes(made):
    """n = 64 as a dense stream is the packed store, whose output may lie on 8 bytes."""
    import torch

    F, G = made[64]
    for cnt in SIZES[:-1]:
        for off in _offsets(F, cnt):
            buf = torch.full((cnt + 3,), -1, dtype=torch.int64, device="cuda")
            G.store_dense(off, cnt, buf[1:])
            got = buf.cpu().numpy().view(np.uint64)
            assert np.array_equal(got[1: cnt + 1], oc.window(F, off, cnt)[:, 0]), (off, cnt)
            assert got[0] == got[cnt + 1] == np.uint64(0xFFFFFFFFFFFFFFFF), (off, cnt)


def test_many_windows(made):
    import torch

    m = hlf.hlf_many_create(400)
    hs, offs, cnts, outs, want = [], [], [], [], []
    for n, (F, G) in made.items():
        for k, cnt in enumerate(SIZES[:-1]):
            o = _offsets(F, cnt)
            off = o[k % len(o)]
            hs.append(G.h)
            offs.append(off)
            cnts.append(cnt)
            outs.append(torch.full((cnt + 2, F.W), -1, dtype=torch.int64, device="cuda"))
            want.append(oc.window(F, off, cnt))
    hlf.hlf_enumerate_store_many(m, hs, offs, cnts, outs)
    torch.cuda.synchronize()
    for off, cnt, o, w in zip(offs, cnts, outs, want):
        got = o.cpu().numpy().view(np.uint64)
        assert np.array_equal(got[:cnt], w), (off, cnt, w.shape)
        assert np.all(got[cnt:] == np.uint64(0xFFFFFFFFFFFFFFFF)), (off, cnt)
    hlf.hlf_many_destroy(m)
