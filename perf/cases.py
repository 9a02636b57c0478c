"""Performance cases of the gs-SGD compression library: what a training program has it do.

A case is one pass through public calls of ``paper_2108_06004_gb300`` on the GPU: a whole
compression step (direct calls, a captured plan, gradients on the host, workers streamed in
batches, one sketch per worker), the step's variants (weight update, HEAVYMIX selection, momentum
and error kept as sketches), and the query alone.

Inputs.  Momentum, error and gradients are normal or Laplace entries with a scale per parameter
block, drawn log-uniform over three decades, plus a few persistent heavy coordinates, as the
library's workloads have them.  All entries lie on a fixed-point grid (as gradients unscaled from a
loss-scaled half-precision backward do) that is coarse enough for every sum of a sketch cell to be
exact in fp32: the cells are updated by atomic additions in no fixed order, and on this grid every
order gives the same cells, hence the same selection.  The momentum factor is 7/8 for the same
reason (0.875 is exact in binary).
"""

import math

import torch

import paper_2108_06004_gb300 as gs

RHO = 0.875
LR = 0.0078125
GRID = 2.0 ** -18          # gradients and error are multiples of this, momentum of 8 times this
P61 = (1 << 61) - 1
MASK64 = (1 << 64) - 1
DEV = "cuda"


def listed():
    return [
        # the smallest call: a small model's gradient, one direct call per step; launches count
        dict(name="step-100k-direct", kind="step", P=4, d=100_003, r=5, c=4096, k=100, dist="normal", plan=False,
             est=False, train=False),
        # d = 2^20 with four workers, captured once and replayed: latency of the whole chain
        dict(name="step-1m-plan", kind="step", P=4, d=1 << 20, r=5, c=1 << 14, k=1000, dist="normal", plan=True,
             est=False, train=False),
        # an odd shape: c not a power of two, even r, five workers, ragged d, the estimate returned
        dict(name="step-3m-odd", kind="step", P=5, d=3_000_017, r=4, c=30_011, k=3000, dist="laplace", plan=False,
             est=True, train=False),
        # ResNet-18-sized training step with the weight update
        dict(name="train-resnet18-plan", kind="step", P=8, d=11_173_962, r=5, c=1 << 17, k=11_200, dist="normal",
             plan=True, est=False, train=True),
        # ResNet-50-sized step: the headline workload
        dict(name="step-resnet50-plan", kind="step", P=8, d=25_557_032, r=5, c=1 << 18, k=25_600, dist="laplace",
             plan=True, est=False, train=False),
        # VGG-16-sized step: sixteen workers, tables larger than L2
        dict(name="step-vgg16-plan", kind="step", P=16, d=138_357_544, r=7, c=1 << 20, k=138_000, dist="normal",
             plan=True, est=False, train=False),
        # BERT-large's sketch with the workers inserted eight at a time, on a quarter of its length
        dict(name="streamed-bert-quarter", kind="streamed", P=16, batch=8, d=83_311_104, r=5, c=1 << 21, k=85_000,
             dist="normal"),
        # the selection the paper prints, at ResNet-50 size
        dict(name="heavymix-resnet50-plan", kind="heavymix", P=8, d=25_557_032, r=5, c=1 << 18, k=25_600,
             dist="laplace", plan=True),
        # momentum and error kept as sketches, at ResNet-50 size
        dict(name="sketched-resnet50-plan", kind="sketched", P=8, d=25_557_032, r=5, c=1 << 18, k=25_600,
             dist="laplace", plan=True),
        # gradients in pinned host memory, results back in host memory, synchronous
        dict(name="host-4m", kind="host", P=4, d=4_194_309, r=5, c=1 << 16, k=4200, dist="normal"),
        # one sketch per worker, each step of the method its own call, no caller workspace
        dict(name="separate-resnet18", kind="separate", P=4, d=11_173_962, r=5, c=1 << 17, k=11_200, dist="normal"),
        # a server that holds a merged sketch: every estimate and the top-k of it
        dict(name="query-resnet50-est", kind="query", P=1, d=25_557_032, r=5, c=1 << 18, k=25_600, dist="laplace",
             est=True),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "streamed", "heavymix", "sketched", "host", "separate", "query"])
    P = {"streamed": rng.choice([9, 12, 16, 24]), "separate": rng.randint(1, 6), "host": rng.randint(1, 8),
         "query": 1}.get(kind) or rng.choice([1, 2, 3, 4, 5, 8, 8, 8, 11, 16])
    d_max = min(138_357_544, 1_200_000_000 // P)
    if kind in ("host", "separate"):
        d_max = min(d_max, 40_000_000 // P) if kind == "host" else min(d_max, 60_000_000)
    d = int(_log_uniform(rng, 70_000, d_max))
    if rng.random() < 0.25:
        d &= ~3
    r = rng.choice([3, 4, 5, 5, 5, 7, 9])
    c = d / _log_uniform(rng, 24, 200)
    if rng.random() < 0.2 and c < 300_000:
        c = max(int(c) | 1, 257)
    else:
        c = 1 << max(8, min(21, int(round(math.log2(c)))))
    k = max(1, int(d * _log_uniform(rng, 3e-4, 4e-3)))
    case = dict(kind=kind, P=P, d=d, r=r, c=c, k=k, dist=rng.choice(["normal", "laplace"]))
    if kind == "streamed":
        case["batch"] = 8
    if kind == "step":
        case.update(plan=rng.random() < 0.6, est=rng.random() < 0.25, train=rng.random() < 0.4)
    if kind in ("heavymix", "sketched"):
        case["plan"] = rng.random() < 0.6
    if kind == "query":
        case["est"] = rng.random() < 0.5
    return case


# ---- inputs --------------------------------------------------------------------------------

class _Sketch:
    """A sketch set that is destroyed with the last reference to it."""

    def __init__(self, r, c, seed, workers, group_width=0):
        self.handle = None
        self.handle = gs.gs_sketch_create(r, c, seed, workers, group_width)

    def __del__(self):
        if self.handle:
            gs.gs_sketch_destroy(self.handle)


class _Table:
    """The merged table of a sketch, as a tensor's array interface."""

    def __init__(self, sketch, shape):
        ptr = gs.gs_sketch_merged_table(sketch.handle)
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False), "version": 3}


def _table(sketch, r, c):
    t = torch.as_tensor(_Table(sketch, (r, c)), device=DEV)
    t.sketch = sketch  # the tensor views the sketch's memory: it keeps the sketch
    return t


def _hash_seed(seed):
    return (seed * 0x9E3779B97F4A7C15 + 12345) & MASK64


def _fill_seed(seed):
    return (seed * 0xD1342543DE82EF95 + 99) & MASK64


def _scales(case, gen):
    """Scale of every coordinate: parameter blocks of uneven sizes, log-uniform scales."""
    d = case["d"]
    top = min(1e-2, 0.2 / math.sqrt(case["P"] * max(1.0, d / case["c"])))
    n = max(1, min(128, d // 500))
    cuts = torch.rand(n, generator=gen, device=DEV).square_().cumsum(0)
    edge = (cuts / cuts[-1] * d).long()
    edge[-1] = d
    s = top * torch.exp(torch.rand(n, generator=gen, device=DEV) * math.log(1e-3))
    return torch.repeat_interleave(s, torch.diff(edge, prepend=edge.new_zeros(1)), output_size=d), top


def _fill(row, case, gen, scale, grid, factor):
    """One worker's vector in place: scaled entries rounded to the grid."""
    if case["dist"] == "laplace":
        row.exponential_(1.0, generator=gen)
        row *= torch.empty_like(row).uniform_(-1.0, 1.0, generator=gen).sign_()
    else:
        row.normal_(0.0, 1.0, generator=gen)
    row.mul_(scale).mul_(factor / grid).round_().mul_(grid)


def _inputs(case, seed):
    """Rows of [P, ld] buffers (ld: d rounded up to four, so that every row is 16-byte aligned)."""
    P, d = case["P"], case["d"]
    ld = (d + 3) // 4 * 4
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    scale, top = _scales(case, gen)
    heavy = torch.randint(0, d, (max(1, d // 2000),), generator=gen, device=DEV)
    bump = torch.zeros(d, device=DEV)
    bump[heavy] = round(4 * top / GRID) * GRID
    names = {"sketched": ("grad",), "query": ("grad",)}.get(case["kind"], ("mom", "err", "grad"))
    out = {}
    for name in names:
        buf = torch.zeros(P, ld, device=DEV)
        grid = 8 * GRID if name == "mom" else GRID
        for p in range(P):
            _fill(buf[p, :d], case, gen, scale, grid, 1.0)
            if name == "grad":
                buf[p, :d] += bump
        out[name] = buf
    if case.get("train") or case["kind"] in ("sketched", "separate"):
        w = torch.empty(d, device=DEV)
        w.normal_(0.0, 0.05, generator=gen)
        out["weights"] = w
    return out


class _State:
    """One program's buffers, sketches and plan (the plan goes first: it names the others)."""

    def __init__(self):
        self.plan = None

    def __del__(self):
        if self.plan:
            gs.gs_plan_destroy(self.plan)


def prepare(case, seed):
    kind, P, d, r, c, k = (case[n] for n in ("kind", "P", "d", "r", "c", "k"))
    s = _State()
    s.kind, s.P, s.d, s.k = kind, P, d, k
    s.inputs = x = _inputs(case, seed)
    rows = lambda name: [x[name][p, :d] for p in range(P)]  # noqa: E731
    hs, s.fill = _hash_seed(seed), _fill_seed(seed)
    s.grad = rows("grad")
    if "mom" in x:
        s.mom, s.err = rows("mom"), rows("err")
    s.weights = x.get("weights")
    s.idx = torch.empty(k, dtype=torch.int64, device=DEV)
    s.vals = torch.empty(k, device=DEV)
    s.est = torch.empty(d, device=DEV) if case.get("est") or kind == "separate" else None

    def ws(nbytes):
        return torch.empty(nbytes, dtype=torch.uint8, device=DEV)

    s.out = {"idx": s.idx}
    if kind != "query":
        s.out["vals"] = s.vals
    if "mom" in x:
        s.out.update(momentum=x["mom"][:, :d], error=x["err"][:, :d])
    if s.est is not None:
        s.out["est"] = s.est
    if s.weights is not None:
        s.out["weights"] = s.weights
    if kind == "separate":
        s.owned = [_Sketch(r, c, hs, 1) for _ in range(P)]
        s.sketches = [o.handle for o in s.owned]
        return s
    s.owned = [_Sketch(r, c, hs, P, case.get("batch", 0))]  # a batch is one group of workers
    if kind == "sketched":
        s.owned += [_Sketch(r, c, hs, 1) for _ in range(2)]
    s.sketches = [o.handle for o in s.owned]
    sk = s.sketches[0]
    if kind == "step":
        s.ws = ws(gs.gs_step_workspace_size(d, k))
        if case["plan"]:
            s.plan = gs.gs_step_plan_create(sk, s.mom, s.err, s.grad, d, RHO, k, s.idx, s.vals, s.est, s.weights, LR,
                                            s.ws)
    elif kind == "streamed":
        s.batch = case["batch"]
        s.ws = ws(gs.gs_query_topk_workspace_size(d, k))
    elif kind == "heavymix":
        s.ws = ws(gs.gs_heavymix_step_workspace_size(d, k))
        s.l2sq = torch.empty(1, dtype=torch.float64, device=DEV)
        s.out["l2sq"] = s.l2sq
        if case["plan"]:
            s.plan = gs.gs_heavymix_step_plan_create(sk, s.mom, s.err, s.grad, d, RHO, k, s.fill, s.idx, s.vals,
                                                     s.l2sq, s.ws)
    elif kind == "sketched":
        s.ws = ws(gs.gs_step_workspace_size(d, k))
        s.out.update(momentum=_table(s.owned[1], r, c), error=_table(s.owned[2], r, c))
        if case["plan"]:
            s.plan = gs.gs_sketched_state_plan_create(sk, s.sketches[1], s.sketches[2], s.grad, d, RHO, k, s.idx,
                                                      s.vals, s.weights, LR, s.ws)
    elif kind == "host":
        s.grad_host = [torch.empty(d, pin_memory=True).copy_(g) for g in s.grad]
        s.idx_host = torch.empty(k, dtype=torch.int64, pin_memory=True)
        s.vals_host = torch.empty(k, pin_memory=True)
        s.ws = ws(gs.gs_step_workspace_size(d, k))
        s.out.update(idx=s.idx_host, vals=s.vals_host)
    elif kind == "query":
        gs.gs_sketch_insert(sk, 0, s.grad[0], d)
        gs.gs_sketch_merge_tree(sk, 1)
        s.ws = ws(gs.gs_query_topk_workspace_size(d, k))
    return s


def run(s):
    d, k = s.d, s.k
    sk = s.sketches[0]
    if s.plan:
        gs.gs_plan_launch(s.plan)
    elif s.kind == "step":
        if s.weights is not None:
            gs.gs_train_step(sk, s.weights, LR, s.mom, s.err, s.grad, d, RHO, k, s.idx, s.vals, s.est, s.ws)
        else:
            gs.gs_step(sk, s.mom, s.err, s.grad, d, RHO, k, s.idx, s.vals, s.est, s.ws)
    elif s.kind == "streamed":
        gs.gs_sketch_zero(sk)
        for p in range(0, s.P, s.batch):
            q = min(p + s.batch, s.P)
            gs.gs_accumulate_insert(sk, p, s.mom[p:q], s.err[p:q], s.grad[p:q], d, RHO)
        gs.gs_sketch_merge_tree(sk, s.P)
        gs.gs_query_topk(sk, d, k, s.idx, None, s.ws)
        gs.gs_gather_and_zero(s.mom, s.err, d, s.idx, k, s.vals)
    elif s.kind == "heavymix":
        gs.gs_heavymix_step(sk, s.mom, s.err, s.grad, d, RHO, k, s.fill, s.idx, s.vals, s.l2sq, s.ws)
    elif s.kind == "sketched":
        gs.gs_sketched_state_step(sk, s.sketches[1], s.sketches[2], s.grad, d, RHO, k, s.idx, s.vals, s.weights, LR,
                                  s.ws)
    elif s.kind == "host":
        gs.gs_step_host(sk, s.mom, s.err, s.grad_host, s.grad, d, RHO, k, s.idx_host, s.vals_host, s.ws)
    elif s.kind == "separate":
        for p in range(s.P):
            gs.gs_accumulate(s.mom[p], s.err[p], s.grad[p], d, RHO)
            gs.gs_sketch_zero(s.sketches[p])
            gs.gs_sketch_insert(s.sketches[p], 0, s.err[p], d)
        gs.gs_sketch_merge_sketches(s.sketches)
        gs.gs_query_topk_noalloc(sk, d, k, s.idx, s.est)
        gs.gs_gather_and_zero(s.mom, s.err, d, s.idx, k, s.vals)
        gs.gs_apply_update(s.weights, d, s.idx, s.vals, k, LR)
    elif s.kind == "query":
        gs.gs_query_topk(sk, d, k, s.idx, s.est, s.ws)
    return s.out


def work(case):
    """Bytes: gradients read once, momentum and error read and written once, the k indices and values
    out, and what else the call returns.  The sketch tables are intermediate except where they are the
    call's input or state.  Operations: three per accumulated entry, one signed addition per sketch row
    and entry, one comparison per row and estimate."""
    kind, P, d, r, c, k = (case[n] for n in ("kind", "P", "d", "r", "c", "k"))
    out = 12 * k + (4 * d if case.get("est") or kind == "separate" else 0) + (8 * k if case.get("train") else 0)
    if kind == "query":
        return {"bytes": 4 * r * c + 4 * d * bool(case.get("est")) + 8 * k, "flops": d * r}
    if kind == "sketched":
        return {"bytes": 4 * P * d + 16 * r * c + out + 8 * k, "flops": P * d * r + d * r}
    return {"bytes": 20 * P * d + out, "flops": P * d * (3 + r) + d * r}


# ---- the same in 64 bits ---------------------------------------------------------------------

def _splitmix(state):
    while True:
        state = (state + 0x9E3779B97F4A7C15) & MASK64
        z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
        yield z ^ (z >> 31)


def _fold(x):
    return (x & P61) + (x >> 61)


def _affine(a, b, i):
    """(a i + b) mod (2^61 - 1) for an int64 tensor i < 2^31."""
    t = (a >> 31) * i
    s = _fold((t >> 30) + ((t & ((1 << 30) - 1)) << 31)) + _fold((a & ((1 << 31) - 1)) * i)
    s = _fold(_fold(s) + b)
    return torch.where(s >= P61, s - P61, s)


_CHUNK = 1 << 24


class _Sketch64:
    def __init__(self, r, c, seed):
        g = _splitmix(seed)
        self.r, self.c = r, c
        self.rows = []
        for _ in range(r):
            a, b, a2, b2 = (next(g) for _ in range(4))
            self.rows.append((1 + a % (P61 - 1), b % P61, 1 + a2 % (P61 - 1), b2 % P61))

    def hash(self, j, i):
        a, b, a2, b2 = self.rows[j]
        return _affine(a, b, i) % self.c, (1 - 2 * (_affine(a2, b2, i) & 1)).double()

    def insert(self, T, at, v, scale=1.0):
        """T += scale * S(v); `at`: the entries' coordinates, or None for all of them in order."""
        for lo in range(0, v.numel(), _CHUNK):
            hi = min(lo + _CHUNK, v.numel())
            i = at[lo:hi] if at is not None else torch.arange(lo, hi, device=DEV)
            for j in range(self.r):
                b, s = self.hash(j, i)
                T[j].index_add_(0, b, s * v[lo:hi] * scale)

    def query(self, T, at, n):
        est = torch.empty(n, dtype=torch.float64, device=DEV)
        step = _CHUNK // 2
        for lo in range(0, n, step):
            hi = min(lo + step, n)
            i = at[lo:hi] if at is not None else torch.arange(lo, hi, device=DEV)
            v = torch.empty(self.r, hi - lo, dtype=torch.float64, device=DEV)
            for j in range(self.r):
                b, s = self.hash(j, i)
                v[j] = s * T[j][b]
            v = v.sort(dim=0).values
            h = self.r // 2
            est[lo:hi] = v[h] if self.r % 2 else 0.5 * (v[h - 1] + v[h])
        return est


def _largest(key, k):
    """Ascending indices of the k largest keys, ties to the smaller index."""
    tau = torch.topk(key, k).values[-1]
    take = key > tau
    eq = (key == tau).nonzero().flatten()[: k - int(take.sum())]
    take[eq] = True
    return take.nonzero().flatten()


def _xi(seed, n):
    """The top 31 bits of the first n splitmix64 outputs of `seed`, as doubles."""
    signed = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731
    shr = lambda z, b: (z >> b) & ((1 << (64 - b)) - 1)  # noqa: E731
    z = torch.arange(1, n + 1, device=DEV) * signed(0x9E3779B97F4A7C15) + signed(seed)
    z = (z ^ shr(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * signed(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 33).double()


def exact(case, seed):
    kind, P, d, r, c, k = (case[n] for n in ("kind", "P", "d", "r", "c", "k"))
    x = _inputs(case, seed)
    sk = _Sketch64(r, c, _hash_seed(seed))
    T = torch.zeros(r, c, dtype=torch.float64, device=DEV)
    total = torch.zeros(d, dtype=torch.float64, device=DEV)
    out = {"idx": None}
    if "mom" in x:
        u, e = (torch.empty(P, d, dtype=torch.float64, device=DEV) for _ in range(2))
        for p in range(P):
            u[p] = x["mom"][p, :d].double() * RHO + x["grad"][p, :d].double()
            e[p] = x["err"][p, :d].double() + u[p]
            total += e[p]
        out.update(momentum=u, error=e)
    else:
        for p in range(P):
            total += x["grad"][p, :d].double()
    w = x.get("weights")
    del x
    sk.insert(T, None, total)
    est = sk.query(T, None, d)
    if case.get("est") or kind == "separate":
        out["est"] = est
    if kind == "query":
        return out
    key = est.abs()
    if kind == "heavymix":
        l2 = (T * T).sum(1).sort().values
        l2 = l2[r // 2] if r % 2 else 0.5 * (l2[r // 2 - 1] + l2[r // 2])
        out["l2sq"] = l2.reshape(1)
        key = torch.where(est * est >= l2 / k, 2.0 ** 32 + key, 2.0 ** 31 - _xi(_fill_seed(seed), d))
    at = _largest(key, k)
    if kind == "sketched":
        vals = est[at]
        U = T.clone()
        sk.insert(T, at, vals, -1.0)
        sk.insert(U, at, sk.query(U, at, k), -1.0)
        out.update(momentum=U, error=T)
    else:
        vals = total[at]
        u[:, at] = 0.0
        e[:, at] = 0.0
    out["vals"] = vals
    if w is not None:
        w = w.double()
        w[at] -= LR * vals
        out["weights"] = w
    return out
