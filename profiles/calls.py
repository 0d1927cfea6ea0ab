"""One small call of each kernel, for a profiler: python profiles/calls.py <case>.

The case's call runs twice (the first loads the code), then the device is waited for.
No case holds more than about 3 GB on the device.
"""

import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import torch  # noqa: E402

import paper_2103_00693_gb300 as hlf  # noqa: E402
import synth  # noqa: E402
from paper_2103_00693_gb300.batch import Batch  # noqa: E402
from synth import workloads  # noqa: E402


def _fac(A):
    f = hlf.Factorization.from_dense(A)
    f.rank
    return f


def _u64(*shape):
    return torch.empty(shape, dtype=torch.int64, device="cuda")


def region():
    f, red = _fac(workloads.grid6()), _u64(hlf.REDUCE_WORDS)
    return lambda: f.reduce(0, 1 << 34, red)


def reduce4():
    f, red = _fac(synth.grid_instance(16, 0.5, 1)), _u64(hlf.REDUCE_WORDS)
    return lambda: f.reduce(0, 1 << 27, red)


def store1():
    f, out = _fac(workloads.grid6()), _u64(1 << 27, 1)
    return lambda: f.store(0, 1 << 27, out)


def dense3():
    f, out = _fac(synth.grid_instance(10, 0.5, 1)), _u64(hlf.dense_words(1 << 25, 100))
    return lambda: f.store_dense(0, 1 << 25, out)


def hist():
    f, out = _fac(synth.grid_instance(8, 0.5, 0)), _u64(1 << 14)
    return lambda: f.histogram(0, 1 << 30, 25, 14, out)


def sample():
    f, out = _fac(synth.grid_instance(8, 0.5, 0)), _u64(1 << 20, 1)
    idx = torch.randint(0, 1 << 30, (1 << 20,), dtype=torch.int64, device="cuda")
    return lambda: f.sample(idx, out)


def _factor(side):
    A = synth.grid_instance(side, 0.5, 1)
    words = torch.from_numpy(hlf.pack_rows(A).view("int64")).cuda()
    return lambda: hlf.Factorization(words, A.shape[0]).close()


def batch():
    B = Batch(workloads.batch()[:1024])
    return lambda: B.run(1 << 20)


CASES = {"region": region, "reduce4": reduce4, "store1": store1, "dense3": dense3, "hist": hist, "sample": sample,
         "factor6": lambda: _factor(6), "factor10": lambda: _factor(10), "factor16": lambda: _factor(16),
         "factor32": lambda: _factor(32), "batch": batch}

if __name__ == "__main__":
    call = CASES[sys.argv[1]]()
    for _ in range(2):
        call()
    torch.cuda.synchronize()
    print(sys.argv[1], "done")
