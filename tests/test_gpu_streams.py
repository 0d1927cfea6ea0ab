"""Calls on different streams side by side: what waits for a factorisation must not
keep another stream's kernels from the SMs."""

import pytest

import paper_2103_00693_gb300 as hlf
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60, 250])
def test_a_reduce_ends_before_the_factorisation_it_runs_beside(cuda_ok, n):
    """A factorisation of n = 1024 keeps one SM for about 200 us and its second launch
    the others for less than 10; a reduce of 20 us that begins 20 us into it is done
    long before it. While the second launch's CTAs sat on every SM from the start, the
    reduce (whole SMs a CTA) ended after it."""
    import torch

    A = torch.from_numpy(hlf.pack_rows(synth.random_symmetric(1024, 0.5, 5)).view("int64")).cuda()
    G = hlf.Factorization.from_dense(synth.random_symmetric(n, 0.5, 1))
    assert G.rank > 30
    side, red = torch.cuda.Stream(), torch.empty(hlf.REDUCE_WORDS, dtype=torch.int64, device="cuda")
    main = torch.cuda.Stream()
    ahead = []
    for _ in range(6):  # the first is a warm-up
        torch.cuda.synchronize()
        start, done, reduced = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        torch.cuda._sleep(4_000_000)  # both streams' work is queued behind it
        start.record()
        main.wait_event(start)
        side.wait_event(start)
        F = hlf.Factorization(A, 1024, main)
        done.record(main)
        with torch.cuda.stream(side):
            torch.cuda._sleep(40_000)
            G.reduce(0, 1 << 20, red, side)
            reduced.record(side)
        torch.cuda.synchronize()
        ahead.append(reduced.elapsed_time(done) * 1e3)
        F.close()
    G.close()
    assert sorted(ahead[1:])[2] > 50, ahead  # us, the median
