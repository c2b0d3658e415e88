"""The contractions whose speed is measured: what they stand for, their inputs, one pass of each
through the public entry points, and the same results in plain 64-bit torch.

A case's tensors are COO lists on the GPU. Their pattern is drawn once for the case; a seed
renames the indices of every mode (paired modes alike) and draws the values, uniform in [-1, 1]
without zeros. So every seed gives other coordinates and other values, and the same number of
products and outputs. Lengths, entry counts and pairings are those of the repository's workloads
and of its tests, and `draw` spreads them over the ranges in between.
"""
import math
import zlib

import numpy as np
import torch

import paper_2410_10094_gb300 as stc

DEVICE = "cuda"


def listed():
    return [
        # The smallest call in ordinary use: two order-3 tensors of 5,000 distinct entries. Latency.
        {"name": "small_64", "path": "contract", "x": "64,64,64", "y": "64,64,64", "cx": "2", "cy": "0",
         "nx": 5000, "ny": 5000, "coords": "distinct"},
        # The large single contraction: order 4, 5e6 uniform entries each, 3.65e8 outputs.
        {"name": "large_256", "path": "contract", "x": "256,256,256,256", "y": "256,256,256,256", "cx": "2,3",
         "cy": "0,1", "nx": 5000000, "ny": 5000000, "coords": "uniform"},
        # A long X against a short, skewed Y: almost every X entry meets nothing.
        {"name": "skewed_y", "path": "contract", "x": "4096,512,512", "y": "512,512,64", "cx": "1,2", "cy": "0,1",
         "nx": 20000000, "ny": 20000, "coords": "zipf_y"},
        # Both operands skewed alike: 2e10 products on 262,144 outputs, all of it multiply and add.
        {"name": "skewed_both", "path": "contract", "x": "4096,512,512", "y": "512,512,64", "cx": "1,2", "cy": "0,1",
         "nx": 20000000, "ny": 20000, "coords": "zipf_both"},
        # The large request of a served mix: order 4, 1e6 entries, two crossed pairs of modes.
        {"name": "middle_128", "path": "contract", "x": "128,128,128,128", "y": "128,128,128,128", "cx": "3,0",
         "cy": "1,2", "nx": 1000000, "ny": 1000000, "coords": "uniform"},
        # A tensor with itself: short ragged modes, order-6 outputs, 2.3e8 of them.
        {"name": "hubbard_1d_p", "path": "contract", "x": "4,4,93,36,432", "y": "", "cx": "1,2", "cy": "1,2",
         "nx": 300000, "ny": 300000, "coords": "self"},
        # Decimal lengths, operands of different order, order-5 outputs, 2.5e7 of them.
        {"name": "set2_ab", "path": "contract", "x": "100,100,100,100,100", "y": "100,100,100,100", "cx": "1,2",
         "cy": "1,2", "nx": 500000, "ny": 500000, "coords": "uniform"},
        # Very sparse: far more contract keys and free keys than entries, about one product each.
        {"name": "nips", "path": "contract", "x": "2000,3000,14000,17000", "y": "", "cx": "1,2", "cy": "1,2",
         "nx": 3000000, "ny": 3000000, "coords": "self"},
        # A contract key space too wide to count in directly (1.2e8), so that its keys are numbered first.
        {"name": "facebook", "path": "contract", "x": "63891,63890,1847", "y": "", "cx": "1,2", "cy": "1,2",
         "nx": 738000, "ny": 738000, "coords": "self"},
        # A chain of two contractions, the first result handed over in key form.
        {"name": "chain_100", "path": "chain", "length": 100, "n1": 200000, "n2": 200000, "n3": 200000},
        # A prepared batch of uneven order-3 pairs (1e2 to 1e5 entries each, lengths 16 to 512), run again and again.
        {"name": "batch_256", "path": "batch", "problems": 256, "sizes": 4},
        # A burst of requests to the server: four small pairs of the batch's mix to one of the order-4 pairs.
        {"name": "serve_20", "path": "serve", "requests": 20, "sizes": 5},
    ]


def draw(rng):
    """One more case: a kind, then its sizes over the range that the listed ones span."""

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def text(v):
        return ",".join(str(int(i)) for i in v)

    kind = rng.choice(["uniform", "uniform", "zipf_y", "zipf_both", "self", "sparse", "chain", "batch", "serve"])
    if kind == "uniform":
        m = rng.choice([1, 2])
        ox, oy = rng.choice([(3, 3), (3, 4), (4, 3), (4, 4), (5, 4)])
        cx, cy = rng.sample(range(ox), m), rng.sample(range(oy), m)
        while True:
            xs = [logint(16, 300) for _ in range(ox)]
            ys = [logint(16, 300) for _ in range(oy)]
            for a, b in zip(cx, cy):
                ys[b] = xs[a]
            nx = logint(2e3, 5e6)
            ny = min(5000000, max(2000, logint(nx / 4, nx * 4)))
            products = nx * ny / math.prod(xs[a] for a in cx)
            if products < 3.5e8 and 2 * nx < math.prod(xs) and 2 * ny < math.prod(ys):
                break
        return {"path": "contract", "x": text(xs), "y": text(ys), "cx": text(cx), "cy": text(cy), "nx": nx, "ny": ny,
                "coords": "uniform"}
    if kind in ("zipf_y", "zipf_both"):
        a, b = rng.randint(300, 600), rng.randint(300, 600)
        fx, fy = rng.randint(1000, 5000), rng.randint(16, 64) if rng.random() < 0.7 else rng.randint(65, 300)
        nx = logint(2e5, 2e7 if kind == "zipf_y" else 8e6)
        ny = logint(2e3, 2e4)
        c = {"path": "contract", "x": text([fx, a, b]), "y": text([a, b, fy]), "cx": "1,2", "cy": "0,1", "nx": nx,
             "ny": ny, "coords": kind}
        if kind == "zipf_y" and rng.random() < 0.4:  # the short operand first, its free mode last in the output
            c = {"path": "contract", "x": text([a, b, fy]), "y": text([fx, a, b]), "cx": "0,1", "cy": "1,2", "nx": ny,
                 "ny": nx, "coords": "zipf_x", "out": "1,0"}
        return c
    if kind == "self":  # short ragged modes, few contract keys
        while True:
            xs = [rng.randint(3, 8), rng.randint(3, 8), rng.randint(60, 140), rng.randint(20, 60), rng.randint(60, 550)]
            n = logint(2e4, 3e5)
            if n * n / (xs[1] * xs[2]) < 2.4e8:
                break
        return {"path": "contract", "x": text(xs), "y": "", "cx": "1,2", "cy": "1,2", "nx": n, "ny": n, "coords": "self"}
    if kind == "sparse":  # many more keys than entries
        if rng.random() < 0.5:
            xs = [rng.randint(1500, 2500), logint(2000, 4000), logint(8000, 16000), logint(8000, 18000)]
        else:
            xs = [logint(20000, 70000), logint(20000, 70000), logint(1500, 70000)]
        n = logint(2e4, 3e6)
        return {"path": "contract", "x": text(xs), "y": "", "cx": "1,2", "cy": "1,2", "nx": n, "ny": n, "coords": "self"}
    if kind == "chain":
        length = rng.randint(60, 120)
        n = logint(4e4, 2e5)
        return {"path": "chain", "length": length, "n1": n, "n2": logint(4e4, n), "n3": logint(4e4, n)}
    if kind == "batch":
        return {"path": "batch", "problems": logint(16, 256), "sizes": rng.randint(100, 1 << 20)}
    return {"path": "serve", "requests": logint(4, 20), "sizes": rng.randint(100, 1 << 20)}


# ------------------------------------------------------------------------------ inputs

def ints(text):
    return tuple(int(v) for v in text.split(",")) if text else ()


def generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def pattern_of(case):
    """The generator of a case's pattern: the same for every seed."""
    return generator(zlib.crc32(repr(sorted((k, v) for k, v in case.items() if k != "name")).encode()))


def uniform(shape, n, g):
    cols = [torch.randint(0, s, (n,), dtype=torch.int32, device=DEVICE, generator=g) for s in shape]
    return torch.stack(cols, 1).contiguous()


def distinct(shape, n, g):
    at = torch.randperm(math.prod(shape), device=DEVICE, generator=g)[:n]
    cols = []
    for s in reversed(shape):
        cols.append((at % s).int())
        at = at // s
    return torch.stack(cols[::-1], 1).contiguous()


def skewed(shape, n, modes, rank_to_cell, g, exponent=1.2):
    """Coordinates whose cell over `modes` follows a Zipf law over the cells, in the given order."""
    cells = rank_to_cell.numel()
    cdf = torch.arange(1, cells + 1, dtype=torch.float64, device=DEVICE).pow(-exponent).cumsum(0)
    u = torch.rand(n, dtype=torch.float64, device=DEVICE, generator=g) * cdf[-1]
    cell = rank_to_cell[torch.searchsorted(cdf, u).clamp_(max=cells - 1)]
    coords = uniform(shape, n, g)
    for m in reversed(modes):
        coords[:, m] = (cell % shape[m]).int()
        cell = cell // shape[m]
    return coords


def renaming(shape, g):
    return [torch.randperm(s, device=DEVICE, generator=g).int() for s in shape]


def tensor(shape, coords, names, g):
    """The tensor of a pattern with its indices renamed and values of its own."""
    coords = torch.stack([names[m][coords[:, m].long()] for m in range(len(shape))], 1).contiguous()
    v = torch.rand(coords.shape[0], dtype=torch.float64, device=DEVICE, generator=g) * 2 - 1
    return (shape, coords, torch.where(v == 0, 0.5, v))


def named_pair(xs, xc, ys, yc, cx, cy, g):
    xn, yn = renaming(xs, g), renaming(ys, g)
    for a, b in zip(cx, cy):
        yn[b] = xn[a]
    return tensor(xs, xc, xn, g), tensor(ys, yc, yn, g)


def pair_of(case, seed):
    """(X, Y, cx, cy, out_order) of a single contraction."""
    p, g = pattern_of(case), generator(seed)
    xs, ys, cx, cy, how = ints(case["x"]), ints(case["y"]), ints(case["cx"]), ints(case["cy"]), case["coords"]
    out = ints(case["out"]) if "out" in case else None
    if how == "self":
        X = tensor(xs, uniform(xs, case["nx"], p), renaming(xs, g), g)
        return X, X, cx, cy, out
    if how == "uniform":
        xc, yc = uniform(xs, case["nx"], p), uniform(ys, case["ny"], p)
    elif how == "distinct":
        xc, yc = distinct(xs, case["nx"], p), distinct(ys, case["ny"], p)
    else:
        order = torch.randperm(math.prod(xs[a] for a in cx), device=DEVICE, generator=p)
        xc = skewed(xs, case["nx"], cx, order, p) if how in ("zipf_both", "zipf_x") else uniform(xs, case["nx"], p)
        yc = skewed(ys, case["ny"], cy, order, p) if how in ("zipf_both", "zipf_y") else uniform(ys, case["ny"], p)
    return (*named_pair(xs, xc, ys, yc, cx, cy, g), cx, cy, out)


def small_sizes(r):
    """Sizes of one order-3 pair of the batched mix: (x shape, y shape, cx, cy, nx, ny)."""
    cx, cy = int(r.randint(0, 3)), int(r.randint(0, 3))
    xs, ys = [int(v) for v in r.randint(16, 513, 3)], [int(v) for v in r.randint(16, 513, 3)]
    ys[cy] = xs[cx]
    nx, ny = (int(round(math.exp(r.uniform(math.log(1e2), math.log(1e5))))) for _ in range(2))
    return tuple(xs), tuple(ys), (cx,), (cy,), nx, ny


def large_sizes(r):
    """Sizes of one order-4 pair of the served mix."""
    cx, cy = (tuple(int(v) for v in r.permutation(4)[:2]) for _ in range(2))
    return (128,) * 4, (128,) * 4, cx, cy, 1000000, 1000000


def many_sizes(case):
    r = np.random.RandomState(case["sizes"])
    if case["path"] == "batch":
        return [small_sizes(r) for _ in range(case["problems"])]
    return [large_sizes(r) if i % 5 == 4 else small_sizes(r) for i in range(case["requests"])]


def many_of(case, seed):
    p, g = pattern_of(case), generator(seed)
    return [(*named_pair(xs, uniform(xs, nx, p), ys, uniform(ys, ny, p), cx, cy, g), cx, cy)
            for xs, ys, cx, cy, nx, ny in many_sizes(case)]


def chain_of(case, seed):
    """A, B, C of (A (x) B) (x) C, modes (2, 3) of the left with (0, 1) of the right each time."""
    p, g, shape = pattern_of(case), generator(seed), (case["length"],) * 4
    names = renaming(shape, g) + renaming(shape, g)
    return [tensor(shape, uniform(shape, case[k], p), n, g)
            for k, n in (("n1", names[:4]), ("n2", names[2:6]), ("n3", names[4:]))]


# ------------------------------------------------------------------------------ one pass

class Served:
    """A running server and its requests; the server stops when the state goes."""

    def __init__(self, requests):
        self.requests = requests
        self.server = stc.Server()

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    if case["path"] == "contract":
        return {"path": "contract", "pair": pair_of(case, seed)}
    if case["path"] == "chain":
        return {"path": "chain", "tensors": chain_of(case, seed)}
    problems = many_of(case, seed)
    if case["path"] == "batch":
        return {"path": "batch", "plan": stc.BatchPlan(problems)}
    return {"path": "serve", "served": Served(problems)}


class Entries(dict):
    """The entries of finished contractions, all of them, for whoever reads them. A contraction's
    result is a set: the library writes it in no particular order, another one on each call. So an
    output that is read here is given in the order of its coordinates; the pass has ended by then,
    and a program that takes the set as it is never comes here."""

    def __init__(self, results):
        super().__init__(coords=None, nnz=None, vals=None)
        self.results = results

    def __getitem__(self, name):
        if name == "nnz":
            return torch.tensor([r.nnz for r in self.results])
        return torch.cat([in_order(r)[name] for r in self.results])


def in_order(r):
    _, where, vals = r.tensor
    if r.keys_form:
        key, at = torch.sort(where)
        return {"coords": key, "vals": vals[at]}
    key = linear(where, r.shape, range(r.order))
    at = torch.sort(key)[1]
    return {"coords": where[at], "vals": vals[at]}


def run(state):
    if state["path"] == "contract":
        X, Y, cx, cy, out = state["pair"]
        return Entries([stc.contract(X, Y, cx, cy, out)])
    if state["path"] == "chain":
        A, B, C = state["tensors"]
        first = stc.contract(A, B, (2, 3), (0, 1), output_keys=True)
        second = stc.contract_keyed(first.tensor, C, (2, 3), (0, 1))
        return {"first": Entries([first]), "second": Entries([second])}
    if state["path"] == "batch":
        return Entries(state["plan"].run())
    served = state["served"]
    tickets = [served.server.submit(*p) for p in served.requests]
    return Entries([served.server.wait(t)[0] for t in tickets])


# ------------------------------------------------------------------------------ the same in plain torch

def linear(coords, shape, modes):
    """Row-major index over the listed modes."""
    key = torch.zeros(coords.shape[0], dtype=torch.int64, device=coords.device)
    for m in modes:
        key = key * int(shape[m]) + coords[:, m]
    return key


def product(X, Y, cx, cy, out=None):
    """(coords, vals, shape) of Z = X (x) Y in the order of its coordinates: every pair of entries
    with equal contract coordinates multiplied, products of equal output coordinates added."""
    (xs, xc, xv), (ys, yc, yv) = X, Y
    xf = [m for m in range(len(xs)) if m not in cx]
    yf = [m for m in range(len(ys)) if m not in cy]
    shape = [xs[m] for m in xf] + [ys[m] for m in yf]
    ky, order = torch.sort(linear(yc, ys, cy))
    fy, yv = linear(yc, ys, yf)[order], yv[order]
    kx, fx = linear(xc, xs, cx), linear(xc, xs, xf)
    lo = torch.searchsorted(ky, kx)
    count = torch.searchsorted(ky, kx, right=True) - lo
    meets = count.nonzero()[:, 0]
    fx, xv, lo, count = fx[meets], xv[meets], lo[meets], count[meets]
    ends = count.cumsum(0)
    total = int(ends[-1]) if ends.numel() else 0
    FY, F = math.prod(ys[m] for m in yf), math.prod(shape)
    dense = F <= 1 << 28
    keys, vals = [], []
    if dense:
        acc = torch.zeros(F, dtype=torch.float64, device=DEVICE)
        seen = torch.zeros(F, dtype=torch.bool, device=DEVICE)
    a, done = 0, 0
    while done < total:
        b = max(a + 1, int(torch.searchsorted(ends, done + (1 << 28), right=True)))
        b = min(b, ends.numel())
        part = count[a:b]
        rows = torch.repeat_interleave(torch.arange(a, b, device=DEVICE), part)
        at = torch.arange(rows.numel(), device=DEVICE) + done
        at = at - (ends[rows] - count[rows]) + lo[rows]
        z = fx[rows] * FY + fy[at]
        v = xv[rows] * yv[at]
        del rows, at
        if dense:
            acc.index_add_(0, z, v)
            seen[z] = True
        else:
            keys.append(z)
            vals.append(v)
        a, done = b, int(ends[b - 1])
    if dense:
        key = seen.nonzero()[:, 0]
        val = acc[key]
    elif keys:
        z, at = torch.sort(torch.cat(keys))
        v = torch.cat(vals)[at]
        new = torch.ones(z.numel(), dtype=torch.bool, device=DEVICE)
        new[1:] = z[1:] != z[:-1]
        key = z[new]
        val = torch.zeros(key.numel(), dtype=torch.float64, device=DEVICE)
        val.index_add_(0, new.long().cumsum(0) - 1, v)
    else:
        key = torch.zeros(0, dtype=torch.int64, device=DEVICE)
        val = torch.zeros(0, dtype=torch.float64, device=DEVICE)
    cols, rest = [], key
    for s in reversed(shape):
        cols.append((rest % s).int())
        rest = rest // s
    coords = torch.stack(cols[::-1], 1) if shape else torch.zeros((key.numel(), 0), dtype=torch.int32, device=DEVICE)
    if out is not None:
        coords, shape = coords[:, list(out)], [shape[q] for q in out]
        at = torch.sort(linear(coords, shape, range(len(shape))))[1]
        coords, val = coords[at], val[at]
    return coords.contiguous(), val, tuple(shape)


def exact(case, seed):
    if case["path"] == "contract":
        coords, vals, _ = product(*pair_of(case, seed))
        return {"coords": coords, "nnz": torch.tensor([vals.numel()]), "vals": vals}
    if case["path"] == "chain":
        A, B, C = chain_of(case, seed)
        coords, vals, shape = product(A, B, (2, 3), (0, 1))
        last, lastv, _ = product((shape, coords, vals), C, (2, 3), (0, 1))
        return {"first": {"coords": linear(coords, shape, range(4)), "nnz": torch.tensor([vals.numel()]), "vals": vals},
                "second": {"coords": last, "nnz": torch.tensor([lastv.numel()]), "vals": lastv}}
    got = [product(*p) for p in many_of(case, seed)]
    return {"coords": torch.cat([g[0] for g in got]), "nnz": torch.tensor([g[1].numel() for g in got]),
            "vals": torch.cat([g[1] for g in got])}


# ------------------------------------------------------------------------------ work and tolerance

def pair_work(xs, ys, cx, cy, nx, ny, how):
    """(bytes read, expected products, expected outputs, bytes of an output) of one contraction."""
    keys = math.prod(xs[m] for m in cx)
    free = math.prod(xs) // keys * (math.prod(ys) // keys)
    products = nx * ny / keys
    read = nx * (4 * len(xs) + 8) + (0 if how == "self" else ny * (4 * len(ys) + 8))
    if how == "zipf_both":
        p = np.arange(1, keys + 1, dtype=np.float64) ** -1.2
        products = nx * ny * float(np.sum((p / p.sum()) ** 2))
    outputs = free * -math.expm1(-products / free)
    if how == "self":  # every entry meets itself, on the diagonal of the output
        side = math.prod(xs) // keys
        outputs += side * -math.expm1(-nx / side)
        products += nx
    return read, products, outputs, 4 * (len(xs) + len(ys) - 2 * len(cx)) + 8


def work(case):
    if case["path"] == "contract":
        xs = ints(case["x"])
        ys = ints(case["y"]) or xs
        parts = [pair_work(xs, ys, ints(case["cx"]), ints(case["cy"]), case["nx"], case["ny"], case["coords"])]
    elif case["path"] == "chain":
        s = (case["length"],) * 4
        r, p, n, each = pair_work(s, s, (2, 3), (0, 1), case["n1"], case["n2"], "uniform")
        parts = [(r, p, n, 16)]  # the result in key form: a 64-bit key and a value
        r, p, n2, each = pair_work(s, s, (2, 3), (0, 1), int(n), case["n3"], "uniform")
        parts.append((int(n) * 16 + case["n3"] * 24, p, n2, each))
    else:
        parts = [pair_work(*q, "uniform") for q in many_sizes(case)]
    return {"bytes": float(sum(r + n * each for r, _, n, each in parts)), "flops": float(sum(2 * p for _, p, _, _ in parts))}


def tolerance(case):
    """Sums of rounded 64-bit products in another order: a few hundred terms in an output at most,
    but for the case where both operands are skewed, which has up to 1e5."""
    if case.get("coords") == "zipf_both":
        return {"rel": 4e-14, "max": 4e-13}
    return {"rel": 1e-15, "max": 2e-14}
