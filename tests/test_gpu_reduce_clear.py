"""Reduces whose result is cleared by the launch before them: into buffers that hold
something, one after another with no wait between, on several streams, and each
followed by a reader on the same stream."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
import synth
from oracle import cpu as oc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 250, 700])
def test_back_to_back(cuda_ok, n):
    import torch

    A = synth.random_symmetric(n, 0.1, n)
    F = oc.factor(A)
    G = hlf.Factorization.from_dense(A)
    # one CTA's worth (nothing to clear), several CTAs, many
    windows = [(5, 100), (3, 70001), (64, 1 << 18), (7, 9), (1, 200003)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    got = []
    for s in streams:
        with torch.cuda.stream(s):
            red = torch.full((hlf.REDUCE_WORDS,), -1, dtype=torch.int64, device="cuda")
            for k in range(12):
                off, cnt = windows[k % len(windows)]
                G.reduce(off, cnt, red)
                got.append((off, cnt, red.clone()))
            parts = torch.full((6, hlf.REDUCE_WORDS), -1, dtype=torch.int64, device="cuda")
            G.reduce_chunks(11, 30000, 6, parts)
            got += [(11 + 30000 * c, 30000, parts[c].clone()) for c in range(6)]
    torch.cuda.synchronize()
    for off, cnt, red in got:
        words = red.cpu().numpy()
        r = hlf.ReduceResult.from_words(words, F.W)
        c, h, f = oc.reduce(F, off, cnt)
        assert (r.count, r.hsum) == (c, h), (off, cnt)
        assert np.array_equal(r.xor_fold, f), (off, cnt)
        assert not words[2 + F.W:].any()
    G.close()
