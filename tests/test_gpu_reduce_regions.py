"""Reduces of at least 2^33 one-word solutions (aligned regions walked over a basis of
their own) against the same windows reduced chunk by chunk, which walk the table's
rows: aligned and ragged windows, both orders, spans with three or more and with
fewer free vectors, and narrow rows that have no high word at all."""

import numpy as np
import pytest

import paper_2103_00693_gb300 as hlf
import synth
from oracle import cpu as oc

pytestmark = pytest.mark.gpu


def _total(parts):
    p = parts.cpu().numpy().view(np.uint64)
    with np.errstate(over="ignore"):
        return [int(p[:, 0].sum(dtype=np.uint64)), int(p[:, 1].sum(dtype=np.uint64))] + \
            np.bitwise_xor.reduce(p[:, 2:], axis=0).tolist()


@pytest.mark.parametrize("order", [hlf.ORDER_GRAY, hlf.ORDER_PAPER])
@pytest.mark.parametrize("name,A", [
    ("grid6", synth.grid_instance(6, 1.0, 3)),
    ("grid6-low", synth.grid_instance(6, 1.0, 1)),
    ("grid8", synth.grid_instance(8, 0.5, 0)),
    ("sym64", synth.random_symmetric(64, 0.5, 3)),
    ("diag34", np.diag([1] * 34).astype(np.uint8)),
])
def test_regions(cuda_ok, name, A, order):
    F = oc.factor(A)
    G = hlf.Factorization.from_dense(A)
    G.set_order(order)
    space = 1 << F.space_log2()
    step = 1 << 26
    for off, k in ((0, 128), (64, 130), (5 << 20, 131), (space - 129 * step, 129), (space // 2 - 100 * step - 3, 256)):
        cnt = k * step
        if off < 0 or off + cnt > space:
            continue
        got = G.reduce(off, cnt).cpu().numpy().view(np.uint64).tolist()
        assert got == _total(G.reduce_chunks(off, step, k)), (name, off, cnt)
    G.close()
