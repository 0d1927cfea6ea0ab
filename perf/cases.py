"""The performance cases of the HLF solver: what a user's program calls, over the
sizes that it calls them with.

A case is a dict with an "op" and its sizes:

    upto     factor one small matrix and store all its solutions up to a cap, with
             one host wait (an interactive or scripted call on a small grid)
    solve    factor, read the rank, store a window of solutions (what one served
             request does)
    stage1   factor and copy the whole factorisation to the host
    reduce   (count, hash sum, XOR-fold) of a window of a resident factorisation,
             in one piece or per chunk, and samples of that window
    store    a window of a resident factorisation as packed words
    dense    the same as a stream of n-bit solutions
    hist     histogram of a bit field over a window
    batch    factor many small grids and reduce each one's first solutions
    many     windows of many resident factorisations in one call (a tick of the
             serving loop)

Matrices are the problem's own: N x N grids whose edges are present with
probability p (p = 1 is the all-connected grid) and whose diagonal is a fair
coin, or symmetric matrices of a given density. Where a window needs a rank,
matrices are redrawn until they have it. Everything the solver returns is made of
whole numbers, so every tolerance is "exact".
"""

import math

import numpy as np
import torch

import paper_2103_00693_gb300 as hlf
from paper_2103_00693_gb300.batch import Batch

GRAY, PAPER = "gray", "paper"


def listed():
    return [
        # the paper's smallest experiment size: every solution of a 3 x 3 grid; all latency
        {"name": "upto_grid3", "op": "upto", "side": 3, "p": 0.5, "cap": 512},
        # a served request of ordinary size: 100 bits, a window at any offset
        {"name": "solve_grid10", "op": "solve", "n": 100, "side": 10, "p": 0.5, "want": 1 << 14, "order": GRAY},
        # a dense matrix with a ragged last word, in the paper's own enumeration order
        {"name": "solve_dense700", "op": "solve", "n": 700, "side": 0, "p": 0.5, "want": 1 << 10, "order": PAPER},
        # stage 1 of the largest grid the solver takes, all of it wanted on the host
        {"name": "stage1_grid32", "op": "stage1", "n": 1024, "side": 32, "p": 0.5},
        # a short reduce of four-word solutions (a spot check, a tail of a job)
        {"name": "reduce_grid16", "op": "reduce", "n": 256, "side": 16, "p": 0.5, "count": (1 << 20) + 4321,
         "chunks": 1, "samples": 0, "order": GRAY},
        # a 2^30 window of a 64-bit grid checked as 64 partial results and 2^20 samples
        {"name": "reduce_grid8_chunks", "op": "reduce", "n": 64, "side": 8, "p": 0.5, "count": 1 << 30,
         "chunks": 64, "samples": 1 << 20, "order": GRAY},
        # full sampling of the all-connected 6 x 6 grid: all solutions of a draw of rank 35
        {"name": "reduce_grid6_all", "op": "reduce", "n": 36, "side": 6, "p": 1.0, "count": 1 << 35,
         "chunks": 1, "samples": 0, "order": GRAY, "whole": True},
        # materialising a window of that grid, a gigabyte at an odd offset
        {"name": "store_grid6", "op": "store", "n": 36, "side": 6, "p": 1.0, "count": (1 << 27) - 77, "order": GRAY},
        # the same as a dense stream where words and solutions do not line up
        {"name": "dense_grid10", "op": "dense", "n": 100, "side": 10, "p": 0.5, "count": (1 << 25) + 19,
         "order": GRAY},
        # an output distribution over 14 bits, as the paper's histograms
        {"name": "hist_grid8", "op": "hist", "n": 64, "side": 8, "p": 0.5, "count": 1 << 30, "bits": 14,
         "order": GRAY},
        # a batch of small grids of mixed sizes
        {"name": "batch_1024", "op": "batch", "grids": 1024, "side_lo": 4, "side_hi": 16, "cap": 1 << 20},
        # one tick of a busy server: 48 windows of all sizes
        {"name": "many_48", "op": "many", "windows": 48, "side_lo": 3, "side_hi": 32, "log2_hi": 18},
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], uniform over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["upto", "solve", "solve", "stage1", "reduce", "reduce", "store", "dense", "hist", "batch", "many"])
    if op == "upto":
        side = rng.randint(2, 8)
        return {"op": op, "side": side, "p": rng.choice([0.5, 1.0]), "cap": _log(rng, 16, 1 << min(side * side, 17))}
    if op == "batch":
        lo = rng.randint(3, 10)
        return {"op": op, "grids": _log(rng, 1, 2048), "side_lo": lo, "side_hi": rng.randint(lo, 16),
                "cap": _log(rng, 1 << 8, 1 << 20)}
    if op == "many":
        lo = rng.randint(3, 16)
        return {"op": op, "windows": _log(rng, 1, 64), "side_lo": lo, "side_hi": rng.randint(lo, 32),
                "log2_hi": rng.randint(11, 19)}
    if op in ("solve", "stage1"):
        if rng.random() < 0.6:
            side = rng.randint(3, 32)
            n, p = side * side, rng.choice([0.5, 0.5, 1.0])
        else:
            side, n, p = 0, _log(rng, 9, 1024), rng.choice([0.5, 0.1])
        c = {"op": op, "n": n, "side": side, "p": p}
        if op == "solve":
            c.update(want=_log(rng, 64, min(1 << 18, 1 << (n // 2 + 2))), order=rng.choice([GRAY, GRAY, PAPER]))
        return c
    # a resident factorisation: grids of every word count, and other symmetric matrices
    if rng.random() < 0.6:
        side = rng.choice([5, 6, 7, 8, 10, 13, 16, 20, 26, 32])
        n, p = side * side, rng.choice([0.5, 1.0])
    else:
        side, n, p = 0, _log(rng, 20, 1024), 0.5
    W = (n + 63) // 64
    c = {"op": op, "n": n, "side": side, "p": p, "order": rng.choice([GRAY, GRAY, GRAY, PAPER])}
    top = (n * 2) // 3  # a rank that most draws have
    if op == "reduce":
        c["chunks"] = rng.choice([1, 1, 1, 7, 64, 1000])
        c["samples"] = rng.choice([0, 0, _log(rng, 1, 1 << 20)])
        c["count"] = c["chunks"] * max(1, _log(rng, 1 << 10, min(1 << top, (1 << 35) // (W * W))) // c["chunks"])
    elif op == "store":
        c["count"] = _log(rng, 1 << 10, min(1 << top, (1 << 27) // W))
    elif op == "dense":
        c["count"] = _log(rng, 1 << 10, min(1 << top, (1 << 32) // n))
    else:
        c["bits"] = rng.randint(4, min(18, n))
        c["count"] = _log(rng, 1 << 10, min(1 << top, 1 << 33))
    return c


# ------------------------------------------------------------------ inputs

def _matrix(rng, n, side, p):
    """A dense 0/1 matrix: a grid of `side` x `side` vertices, or (side 0) a
    symmetric matrix of density p; the grid's diagonal is a fair coin."""
    A = np.zeros((n, n), dtype=np.uint8)
    if side:
        v = np.arange(n).reshape(side, side)
        i = np.concatenate([v[:, :-1].ravel(), v[:-1, :].ravel()])
        j = np.concatenate([v[:, 1:].ravel(), v[1:, :].ravel()])
        keep = rng.random(i.size) < p
        A[i[keep], j[keep]] = A[j[keep], i[keep]] = 1
        A[np.arange(n), np.arange(n)] = rng.random(n) < 0.5
    else:
        U = np.triu((rng.random((n, n)) < p).astype(np.uint8))
        A = U | U.T
    return A


def _ints(A):
    """The rows of A as Python integers, column j at bit j."""
    packed = np.packbits(A, axis=1, bitorder="little")
    return [int.from_bytes(r.tobytes(), "little") for r in packed]


def _reduced(rows, n):
    """(pivot columns, reduced rows) of a 0/1 matrix over the field of two elements."""
    left, piv, out = [r for r in rows if r], [], []
    for c in range(n):
        k = next((k for k, r in enumerate(left) if r >> c & 1), None)
        if k is None:
            continue
        b = left.pop(k)
        left = [x for x in (r ^ b if r >> c & 1 else r for r in left) if x]
        out = [r ^ b if r >> c & 1 else r for r in out]
        piv.append(c)
        out.append(b)
    return piv, out


def _draw_matrix(case, seed, rank=0):
    """A matrix of at least this rank, or of exactly it where the window is the
    whole index space."""
    rng = np.random.Generator(np.random.PCG64(seed))
    for _ in range(4000):
        A = _matrix(rng, case["n"], case["side"], case["p"])
        r = len(_reduced(_ints(A), case["n"])[0]) if rank else 0
        if r == rank or r > rank and not case.get("whole"):
            return A, rng
    raise ValueError("no matrix of rank %d in 4000 draws" % rank)


def _need(case):
    """The rank a case's window needs."""
    return {"solve": case.get("want", 1), "stage1": 1}.get(case["op"], case.get("count", 1)) - 1


def _problem(case, seed):
    """(A, offset, sample indices) of a single-matrix case."""
    A, rng = _draw_matrix(case, seed, _need(case).bit_length())
    u = int(rng.integers(0, 1 << 62))
    idx = rng.integers(0, case["count"], case["samples"]) if case.get("samples") else None
    return A, u, idx


def _offset(u, r, count):
    """Anywhere in the index space, or its start when the window is all of it."""
    return u % ((1 << min(r, 62)) - count + 1)


def _device_rows(A):
    return torch.from_numpy(hlf.pack_rows(A).view(np.int64)).cuda()


def _many(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    got = []
    for k in range(case["windows"]):
        # sides and windows spread alike for every seed, so that a pass is as much work
        part = (k + 0.5) / case["windows"]
        side = case["side_lo"] + round(part * (case["side_hi"] - case["side_lo"]))
        A = _matrix(rng, side * side, side, 0.5)
        lo = min(10, case["log2_hi"])
        got.append((side, A, int(2 ** (lo + (k * 0.618034 % 1) * (case["log2_hi"] - lo))), int(rng.integers(0, 1 << 62))))
    return got


def _many_count(side, want):
    """A window that every draw of a grid of this side has: half its vertices is a
    safe rank from 4 x 4 on; smaller grids give their whole windows away."""
    return min(want, 1 << (side * side // 2)) if side > 3 else 1


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        rng = np.random.Generator(np.random.PCG64(seed))
        sides = np.linspace(case["side_lo"], case["side_hi"], case["grids"]).round().astype(int)
        mats = [_matrix(rng, s * s, s, 0.5) for s in map(int, rng.permutation(sides))]
        return {"op": op, "cap": case["cap"], "batch": Batch(mats)}
    if op == "many":
        facs, offs, counts, words = [], [], [], []
        for side, A, want, u in _many(case, seed):
            f = hlf.Factorization.from_dense(A)
            c = min(_many_count(side, want), 1 << min(f.rank, 62))
            facs.append(f)
            counts.append(c)
            offs.append(_offset(u, f.rank, c))
            words.append(-(-c * f.W // 2) * 2)  # 16-byte aligned blocks
        buf = torch.zeros(sum(words), dtype=torch.int64, device="cuda")
        outs, at = [], 0
        for w in words:
            outs.append(buf[at: at + w])
            at += w
        return {"op": op, "plan": hlf.hlf_many_create(case["windows"]), "facs": facs, "h": [f.h for f in facs],
                "offs": offs, "counts": counts, "outs": outs, "buf": buf}
    if op == "upto":
        A, _ = _draw_matrix({"n": case["side"] ** 2, **case}, seed)
        return {"op": op, "A": _device_rows(A), "n": case["side"] ** 2, "cap": case["cap"],
                "out": torch.zeros((case["cap"], (case["side"] ** 2 + 63) // 64), dtype=torch.int64, device="cuda")}
    A, u, idx = _problem(case, seed)
    n, W = case["n"], (case["n"] + 63) // 64
    s = {"op": op, "n": n, "order": hlf.ORDER_PAPER if case.get("order") == PAPER else hlf.ORDER_GRAY}
    rows = _device_rows(A)
    if op in ("solve", "stage1"):
        s.update(A=rows, u=u, want=case.get("want"))
        if op == "solve":
            s["out"] = torch.zeros((case["want"], W), dtype=torch.int64, device="cuda")
        else:  # the caller's arrays, sized before the rank is known
            s.update(piv=np.full(n, -1, dtype=np.int32), basis=np.zeros((n, W), dtype=np.int64))
        return s
    f = hlf.Factorization(rows, n)
    f.set_order(s["order"])
    count = case["count"]
    s.update(f=f, count=count, offset=_offset(u, f.rank, count))
    if op == "reduce":
        s.update(chunks=case["chunks"], red=torch.zeros((case["chunks"], hlf.REDUCE_WORDS), dtype=torch.int64, device="cuda"))
        s["idx"] = torch.from_numpy(idx + s["offset"]).cuda() if idx is not None else None
        s["smp"] = torch.zeros((idx.size, W), dtype=torch.int64, device="cuda") if idx is not None else None
    elif op == "store":
        s["out"] = torch.zeros((count, W), dtype=torch.int64, device="cuda")
    elif op == "dense":
        s["out"] = torch.zeros(hlf.dense_words(count, n), dtype=torch.int64, device="cuda")
    else:
        s.update(bits=case["bits"], lo=(n - case["bits"]) // 2, out=torch.zeros(1 << case["bits"], dtype=torch.int64, device="cuda"))
    return s


# --------------------------------------------------------------------- run

def run(s):
    op = s["op"]
    if op == "upto":
        f = hlf.Factorization(s["A"], s["n"])
        f.store_upto(s["cap"], s["out"])
        torch.cuda.current_stream().synchronize()  # the caller reads the solutions next
        r = f.rank
        f.close()
        return {"rank": r, "z": s["out"]}
    if op == "solve":
        f = hlf.Factorization(s["A"], s["n"])
        f.set_order(s["order"])
        r = f.rank
        f.store(_offset(s["u"], r, s["want"]), s["want"], s["out"])
        f.close()
        return {"rank": r, "z": s["out"]}
    if op == "stage1":
        f = hlf.Factorization(s["A"], s["n"])
        piv, z0, basis = f.factor_host()
        f.close()
        s["piv"][: piv.size] = piv
        s["basis"][: piv.size] = basis.view(np.int64)
        return {"piv": s["piv"], "z0": z0.view(np.int64), "basis": s["basis"]}
    if op == "batch":
        s["batch"].run(s["cap"])
        return {"rank": s["batch"].r_dev, "red": s["batch"].red_dev}
    if op == "many":
        hlf.hlf_enumerate_store_many(s["plan"], s["h"], s["offs"], s["counts"], s["outs"])
        return s["buf"]
    f = s["f"]
    if op == "reduce":
        if s["chunks"] == 1:
            f.reduce(s["offset"], s["count"], s["red"])
        else:
            f.reduce_chunks(s["offset"], s["count"] // s["chunks"], s["chunks"], s["red"])
        if s["idx"] is None:
            return s["red"]
        return {"red": s["red"], "samples": f.sample(s["idx"], s["smp"])}
    if op == "store":
        return f.store(s["offset"], s["count"], s["out"])
    if op == "dense":
        return f.store_dense(s["offset"], s["count"], s["out"])
    return f.histogram(s["offset"], s["count"], s["lo"], s["bits"], s["out"])


# -------------------------------------------------------------------- work

def work(case):
    """Bytes: each input read once and each output written once. Operations:
    32-bit integer ones, of the elimination (half of n * n row XORs) and of the
    solutions: one row XOR each, and for a reduce the hash's multiplications,
    shifts and additions (22 W - 4 in all)."""
    op = case["op"]
    if op == "batch":
        sides = np.linspace(case["side_lo"], case["side_hi"], case["grids"]).round().astype(int)
        n = sides.astype(float) ** 2
        W = np.ceil(n / 64)
        count = np.minimum(case["cap"], 2.0 ** (n * 0.85))  # ranks are about 0.85 n
        return {"bytes": float((8 * n * W + 148).sum()), "flops": float((n * n * W + (22 * W - 4) * count).sum())}
    if op == "many":
        got = [(math.ceil(side * side / 64), _many_count(side, want)) for side, _, want, _ in _many(case, 0)]
        return {"bytes": float(sum(8 * W * c for W, c in got)), "flops": float(sum(2 * W * c for W, c in got))}
    n = case["side"] ** 2 if op == "upto" else case["n"]
    W = (n + 63) // 64
    if op == "upto":
        return {"bytes": 8.0 * W * (n + case["cap"]), "flops": float(n * n * W + 2 * W * case["cap"])}
    if op == "solve":
        return {"bytes": 8.0 * W * (n + case["want"]), "flops": float(n * n * W + 2 * W * case["want"])}
    if op == "stage1":
        return {"bytes": 16.0 * W * n, "flops": float(n * n * W)}
    c = float(case["count"])
    if op == "reduce":
        m = case["samples"]
        return {"bytes": 8.0 * 66 * W + 144 * case["chunks"] + 8 * m * (1 + W), "flops": (22 * W - 4) * c + 64.0 * W * m}
    if op == "store":
        return {"bytes": 8.0 * W * c, "flops": 2 * W * c}
    if op == "dense":
        return {"bytes": n * c / 8, "flops": 2 * W * c}
    return {"bytes": 8.0 * (66 * W + (1 << case["bits"])), "flops": 2 * c}


def tolerance(case):
    return "exact"


# ------------------------------------------------------------------- exact

def _signed(x):
    return x - (1 << 64) if x >> 63 & 1 else x


class _Plain:
    """The factorisation and its enumeration in plain Python integers and torch."""

    def __init__(self, A, paper=False):
        self.n = A.shape[0]
        self.W = (self.n + 63) // 64
        rows = _ints(A)
        self.piv, self.basis = _reduced(rows, self.n)
        self.r = len(self.piv)
        self.z0 = 0
        for f in sorted(set(range(self.n)) - set(self.piv)):
            x = 1 << f
            for c, b in zip(self.piv, self.basis):
                x |= (b >> f & 1) << c
            q = sum((rows[i] & x).bit_count() for i in range(self.n) if x >> i & 1)
            self.z0 |= (q % 4 // 2) << f
        self.paper = paper
        # the row each bit of the index (paper) or of its Gray code selects
        self.step = [rows[c] for c in reversed(self.piv)] if paper else self.basis

    def word(self, x, w):
        return _signed(x >> 64 * w & (1 << 64) - 1)

    def at(self, idx):
        """The solutions of an int64 tensor of indices, [len(idx)][W]."""
        g = idx if self.paper else idx ^ (idx >> 1)
        z = torch.empty((idx.numel(), self.W), dtype=torch.int64, device=idx.device)
        for w in range(self.W):
            col = torch.full_like(idx, self.word(self.z0, w))
            for k in range(min(self.r, 63)):
                v = self.word(self.step[k], w)
                if v:
                    col ^= -((g >> k) & 1) & v
            z[:, w] = col
        return z

    def blocks(self, offset, count, log2=22):
        """(first index, solutions) of the window, aligned block by block. The
        solutions of a block are those of block 0 with the same word XORed in."""
        size = 1 << log2
        base = self.at(torch.arange(size, dtype=torch.int64, device="cuda"))
        for b in range(offset >> log2, (offset + count - 1 >> log2) + 1):
            lo, hi = max(offset, b << log2), min(offset + count, b + 1 << log2)
            z = base
            if b & 1 and not self.paper:  # the Gray code of an odd block is that of block 0 with its top bit flipped
                z = base ^ torch.tensor([self.word(self.step[log2 - 1], w) for w in range(self.W)], device="cuda")
            g = b if self.paper else b ^ (b >> 1)
            x = 0
            for k in range(g.bit_length()):
                if g >> k & 1:
                    x ^= self.step[log2 + k]
            if x:
                z = z ^ torch.tensor([self.word(x, w) for w in range(self.W)], device="cuda")
            yield lo, z[lo - (b << log2): hi - (b << log2)]


def _shift(x, s):
    return (x >> s) & ((1 << 64 - s) - 1)


def _mix(x):
    x = (x ^ _shift(x, 30)) * _signed(0xBF58476D1CE4E5B9)
    x = (x ^ _shift(x, 27)) * _signed(0x94D049BB133111EB)
    return x ^ _shift(x, 31)


def _fold(z):
    """XOR of the rows of z."""
    while z.shape[0] > 1:
        if z.shape[0] & 1:
            z = torch.cat([z, torch.zeros_like(z[:1])])
        z = z[: z.shape[0] // 2] ^ z[z.shape[0] // 2:]
    return z[0]


def _reduce_of(P, offset, count):
    out = torch.zeros(hlf.REDUCE_WORDS, dtype=torch.int64, device="cuda")
    out[0] = count
    for _, z in P.blocks(offset, count, 22 if count >= 1 << 22 else 12):
        h = _mix(z[:, 0])
        for w in range(1, P.W):
            h = _mix(h ^ z[:, w])
        out[1] += h.sum()
        out[2: 2 + P.W] ^= _fold(z)
    return out


def exact(case, seed):
    op = case["op"]
    if op in ("batch", "many") or case.get("count", 0) * ((case.get("n", 1) + 63) // 64) > 1 << 31 \
            or case.get("chunks", 1) > 64:
        return None
    if op == "upto":
        A, _ = _draw_matrix({"n": case["side"] ** 2, **case}, seed)
        P = _Plain(A)
        z = torch.zeros((case["cap"], P.W), dtype=torch.int64, device="cuda")
        k = min(1 << P.r, case["cap"])
        z[:k] = P.at(torch.arange(k, dtype=torch.int64, device="cuda"))
        return {"rank": P.r, "z": z}
    A, u, idx = _problem(case, seed)
    P = _Plain(A, case.get("order") == PAPER)
    if op == "solve":
        off = _offset(u, P.r, case["want"])
        return {"rank": P.r, "z": P.at(torch.arange(off, off + case["want"], dtype=torch.int64, device="cuda"))}
    if op == "stage1":
        words = [[P.word(b, w) for w in range(P.W)] for b in [P.z0] + P.basis + [0] * (P.n - P.r)]
        words = np.array(words, dtype=np.int64)
        return {"piv": np.array(P.piv + [-1] * (P.n - P.r), dtype=np.int32), "z0": words[0], "basis": words[1:]}
    count = case["count"]
    off = _offset(u, P.r, count)
    if op == "reduce":
        c = count // case["chunks"]
        red = torch.stack([_reduce_of(P, off + k * c, c) for k in range(case["chunks"])])
        return red if idx is None else {"red": red, "samples": P.at(torch.from_numpy(idx + off).cuda())}
    if op == "store":
        return torch.cat([z for _, z in P.blocks(off, count, 22 if count >= 1 << 22 else 12)])
    if op == "hist":
        lo, out = (case["n"] - case["bits"]) // 2, torch.zeros(1 << case["bits"], dtype=torch.int64, device="cuda")
        for _, z in P.blocks(off, count, 22 if count >= 1 << 22 else 12):
            w, b = lo // 64, lo % 64
            v = _shift(z[:, w], b) if b else z[:, w].clone()
            if b and w + 1 < P.W:
                v |= z[:, w + 1] << 64 - b
            out += torch.bincount(v & (1 << case["bits"]) - 1, minlength=out.numel())
        return out
    n, at, out = case["n"], 0, torch.zeros(hlf.dense_words(count, case["n"]), dtype=torch.int64, device="cuda")
    place = torch.tensor([_signed(1 << k) for k in range(64)], device="cuda")
    while at < count:  # 64 solutions fill n words
        m = min(count - at, 1 << 18)
        z = P.at(torch.arange(off + at, off + at + m, dtype=torch.int64, device="cuda"))
        bits = torch.cat([(z[:, w: w + 1] >> torch.arange(min(64, n - 64 * w), device="cuda")) & 1 for w in range(P.W)], 1).reshape(-1)
        bits = torch.nn.functional.pad(bits, (0, -bits.numel() % 64)).reshape(-1, 64)
        out[at * n // 64: at * n // 64 + bits.shape[0]] = (bits * place).sum(1)
        at += m
    return out
