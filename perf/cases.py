"""The calls that this library is measured on: one pass each through its public entry points.

A case is a dict of plain values.  Tensors are column-major in label order, so a tensor with
extents (e0, .., er) is a torch tensor of shape (er, .., e0).  Kinds:

  contract   Plan.contract: one planned expression (two operands or a chain; FP64, split-BF16 or
             emulated-FP64 arithmetic; optionally an operand that is a view of a stored tensor)
  host       Plan.contract_host: the same from pinned host buffers to a pinned host buffer
  backward   autograd.einsum of a three-operand chain and the gradients of all its operands
  copy       transpose: a bit-exact permutation
  batched    BatchedPlan.contract over uneven blocks, reduced in the kernel or stored
  triples    TriplesPlan.energy: nine permuted terms accumulated per block, energies out
"""
import itertools
import math
import random
import re

import numpy as np
import torch

import paper_2102_06827_gb300 as comet
from paper_2102_06827_gb300 import autograd

DTYPES = {"f32": torch.float32, "f64": torch.float64}
BYTES = {"f32": 4, "f64": 8}
PRECISION_DTYPE = {"native": "f64", "split_bf16": "f32", "emu_f64": "f64"}

RANK3 = "C[a,b,c,d] = A[a,e,b] * B[e,d,c]"
RING = "C[i,a,j,b] = A[k,a,c,i] * B[c,b,k,j]"          # the CCSD ring contraction
CHAIN = "D[a,b] = A[a,i,j] * B[i,j,k,l] * C[k,l,b]"
# multi-operand coupled-cluster terms; occupied labels i j m n, virtual labels a .. f
TERMS = ("X[i,a] = A[c,d,m,n] * B[i,n,a,d] * C[m,c]",
         "X[i,a] = A[c,d,m,n] * B[i,d] * C[n,a] * D[m,c]",
         "X[j,i,a,b] = A[m,n,e,j] * B[e,i] * C[a,m] * D[b,n]",
         "X[i,a,b,j] = A[m,n,f,e] * B[e,i] * C[f,n] * D[a,b,m,j]",
         "X[a,b,i,j] = A[m,n,e,f] * B[a,m] * C[f,n] * D[e,b,i,j]")
BLOCK = "T[a,b,c,i,j,k] = A[d,a,b,i] * B[c,d,j,k]"
BLOCK_LABELS = ("a", "b", "c", "i", "j", "k", "d")
SIGNS = (-1, -1, -1, 1, 1, 1)


def listed():
    return [
        # one small tensor contraction in full precision, as a program with many of them calls it:
        # the time is latency
        dict(name="f64_small", kind="contract", expr=RANK3, ext="a=24,b=24,c=24,d=24,e=24", precision="native"),
        # a ring term of a small molecule: launches count more than arithmetic
        dict(name="split_small", kind="contract", expr=RING, ext=_ring(8, 24), precision="split_bf16"),
        # a ring term at an ordinary size that no tile divides
        dict(name="split_odd", kind="contract", expr=RING, ext=_ring(23, 71), precision="split_bf16"),
        # the ring term of the benchmark, the largest call
        dict(name="split_large", kind="contract", expr=RING, ext=_ring(64, 192), precision="split_bf16"),
        # the same term where FP64 results are needed
        dict(name="emulated_f64", kind="contract", expr=RING, ext=_ring(24, 72), precision="emu_f64"),
        # a four-operand term: a tensor-times-matrix step, small GEMMs and a matrix-vector step
        dict(name="chain", kind="contract", expr=TERMS[1], ext=_occ_virt(48, 144), precision="split_bf16"),
        # a training step's forward and backward through a three-operand chain
        dict(name="backward", kind="backward", ab=256, ijkl="48,48,48,48", precision="split_bf16"),
        # a term whose tensors live in host memory
        dict(name="host_ring", kind="host", expr=RING, ext=_ring(40, 120), precision="split_bf16"),
        # reordering a six-index tensor with odd leading extents
        dict(name="copy_f32_odd", kind="copy", dtype="f32", ext="15,30,31,21,31,12", perm="3,0,4,2,1,5"),
        # reordering a large four-index tensor
        dict(name="copy_f64_large", kind="copy", dtype="f64", ext="64,192,64,160", perm="3,1,2,0"),
        # triples blocks of uneven size, consumed as they are formed
        dict(name="batched", kind="batched", blocks=256, lo=8, hi=32, shapes=3, precision="split_bf16", store=False),
        # the triples energy of a batch of blocks
        dict(name="triples", kind="triples", blocks=16, lo=8, hi=32, shapes=3, dtype="f32"),
    ]


def draw(rng):
    kind = rng.choice(["contract"] * 6 + ["host", "backward", "copy", "copy", "copy", "batched", "triples"])
    if kind == "contract":
        which = rng.choice(["rank3", "ring", "ring", "ring", "emulated", "terms"])
        if which == "rank3":
            ext = ",".join(f"{l}={_log(rng, 8, 48)}" for l in "abcde")
            return dict(kind=kind, expr=RANK3, ext=ext, precision="native")
        if which == "terms":
            o = _log(rng, 8, 56)
            return dict(kind=kind, expr=rng.choice(TERMS), ext=_occ_virt(o, _virtuals(rng, o, 168)), precision="split_bf16")
        o = _log(rng, 4, 30 if which == "emulated" else 63)
        case = dict(kind=kind, expr=RING, ext=_ring(o, _virtuals(rng, o, 90 if which == "emulated" else 190)),
                    precision="emu_f64" if which == "emulated" else "split_bf16")
        if which == "ring" and o < 24 and rng.random() < 0.25:
            case["view"] = True
        return case
    if kind == "host":
        o = _log(rng, 8, 40)
        return dict(kind=kind, expr=RING, ext=_ring(o, _virtuals(rng, o, 120)), precision="split_bf16")
    if kind == "backward":
        return dict(kind=kind, ab=_log(rng, 24, 256), ijkl=",".join(str(_log(rng, 8, 48)) for _ in range(4)),
                    precision="split_bf16")
    if kind == "copy":
        dtype, rank = rng.choice(["f32", "f64"]), rng.choice([3, 4, 4, 5, 6, 6])
        while True:
            target = math.exp(rng.uniform(math.log(1 << 20), math.log(1 << 30)))
            ext = [_log(rng, 8, 256) for _ in range(rank - 1)]
            last = round(target / (BYTES[dtype] * math.prod(ext)))
            if 8 <= last <= 256:
                break
        ext.insert(rng.randrange(rank), last)
        perm = list(range(rank))
        while perm == sorted(perm):
            rng.shuffle(perm)
        return dict(kind=kind, dtype=dtype, ext=",".join(map(str, ext)), perm=",".join(map(str, perm)))
    shapes = rng.randrange(1000)
    if kind == "batched":
        store = rng.random() < 0.4
        return dict(kind=kind, blocks=_log(rng, 2, 12) if store else _log(rng, 8, 256), lo=8, hi=rng.choice([12, 16, 24, 32]),
                    shapes=shapes, precision="split_bf16", store=store)
    f64 = rng.random() < 0.3
    return dict(kind=kind, blocks=_log(rng, 2, 10), lo=8, hi=rng.choice([11, 16] if f64 else [16, 24, 32]), shapes=shapes,
                dtype="f64" if f64 else "f32")


def prepare(case, seed):
    return {"contract": _prepare_contract, "host": _prepare_host, "backward": _prepare_backward, "copy": _prepare_copy,
            "batched": _prepare_batched, "triples": _prepare_triples}[case["kind"]](case, _generator(seed))


def run(state):
    return state["call"]()


def work(case):
    kind = case["kind"]
    if kind in ("contract", "host"):
        ext, size = _extents(case["ext"]), BYTES[PRECISION_DTYPE[case["precision"]]]
        elems = sum(math.prod(ext[l] for l in ls) for ls in _labels(case["expr"]))
        return {"bytes": size * elems, "flops": _fewest_flops(case["expr"], ext)}
    if kind == "backward":
        ext = _chain_extents(case)
        names = _labels(CHAIN)
        elems = sum(math.prod(ext[l] for l in ls) for ls in names)
        flops = _fewest_flops(CHAIN, ext)
        for p in range(1, 4):          # the gradient of an operand: the others and the output's gradient onto its labels
            flops += _fewest([names[q] for q in range(4) if q != p], names[p], ext)
        return {"bytes": 4 * 2 * elems, "flops": flops}
    if kind == "copy":
        return {"bytes": 2 * BYTES[case["dtype"]] * math.prod(_ints(case["ext"])), "flops": 0}
    table = _table(case)
    t = np.prod(table[:, :6], axis=1, dtype=np.float64)
    a, b, c, i, j, k, d = table.T.astype(np.float64)
    if kind == "batched":
        out = t.sum() * 4 if case["store"] else 16 * len(table)
        return {"bytes": 4 * float((d * a * b * i + c * d * j * k).sum()) + out, "flops": float(2 * (t * d).sum())}
    elems = sum(float(np.prod([table[:, BLOCK_LABELS.index(l)] for l in ls], axis=0, dtype=np.float64).sum())
                for term in _terms() for ls in _labels(term)[1:])
    return {"bytes": BYTES[case["dtype"]] * elems, "flops": float(18 * (t * d).sum())}


def exact(case, seed):
    g, kind = _generator(seed), case["kind"]
    if kind in ("contract", "host"):
        ins, views = _contract_inputs(case, g)
        ins = [x[v] if v else x for x, v in zip(ins, views)]
        return _contract_exact(case["expr"], [x.double() for x in ins])
    if kind == "backward":
        ops, grad = _chain_inputs(case, g)
        ops = [x.double().requires_grad_(True) for x in ops]
        out = _contract_exact(CHAIN, ops)
        return (out.detach(), *torch.autograd.grad(out, ops, grad.double()))
    if kind == "copy":
        x, ext, perm = _copy_input(case, g)
        r = len(ext)
        return x.double().permute(*[r - 1 - p for p in reversed(perm)]).contiguous()
    table = _table(case)
    if kind == "triples":
        ops, eps = _triples_inputs(case, table, g)
        return torch.stack([_energy_exact(row, o, e) for row, o, e in zip(table, ops, eps)])
    a, b = _batched_inputs(table, g)
    if case["store"]:
        _, offs, total = _packed([math.prod(r[:6]) for r in table.tolist()])
        out = torch.zeros(total, dtype=torch.float64, device="cuda")
        for row, o, x, y in zip(table.tolist(), offs, a, b):
            t = _contract_exact(BLOCK, [x.double(), y.double()])
            out[o:o + t.numel()] = t.reshape(-1)
        return out
    return torch.tensor([v for n, (row, x, y) in enumerate(zip(table.tolist(), a, b)) for v in _sums_exact(n, row, x.double(), y.double())],
                        dtype=torch.float64)


# ---- extents and labels -------------------------------------------------------------------------

def _log(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _virtuals(rng, o, most):
    return min(most, round(o * rng.uniform(2.0, 4.0)))


def _ring(o, v):
    return f"i={o},j={o},k={o},a={v},b={v},c={v}"


def _occ_virt(o, v):
    return ",".join([f"{l}={o}" for l in "ijmn"] + [f"{l}={v}" for l in "abcdef"])


def _ints(text):
    return [int(x) for x in text.split(",")]


def _extents(text):
    return {k: int(v) for k, v in (x.split("=") for x in text.split(","))}


def _labels(expr):
    """Labels of every tensor, the result's first."""
    return [tuple(x.strip() for x in m.split(",")) for m in re.findall(r"\[([^\]]*)\]", expr)]


def _fewest(operands, result, ext):
    """Flops of the cheapest binary contraction order."""
    best = math.inf
    if len(operands) == 1:
        return 0.0
    for p, q in itertools.combinations(range(len(operands)), 2):
        rest = [operands[r] for r in range(len(operands)) if r not in (p, q)]
        kept = set(result).union(*rest)
        both = set(operands[p]) | set(operands[q])
        best = min(best, 2.0 * math.prod(ext[l] for l in both) + _fewest(rest + [tuple(both & kept)], result, ext))
    return best


def _fewest_flops(expr, ext):
    result, *operands = _labels(expr)
    return _fewest(operands, result, ext)


# ---- inputs ---------------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, extents, dtype, scale=1.0):
    """Column-major tensor, uniform in [-scale, scale)."""
    x = torch.rand(tuple(reversed(extents)), generator=g, dtype=dtype, device="cuda")
    return x.mul_(2 * scale).sub_(scale)


def _packed(sizes):
    """(sizes, offsets, total) of arrays that lie one after another, each on 16 bytes."""
    starts = np.concatenate([[0], np.cumsum([(s + 3) // 4 * 4 for s in sizes])])
    return sizes, starts[:-1].tolist(), int(starts[-1])


def _table(case):
    """Extents of the blocks: uniform in lo .. hi, a row for each block."""
    r = random.Random(case["shapes"])
    return np.array([[r.randint(case["lo"], case["hi"]) for _ in BLOCK_LABELS] for _ in range(case["blocks"])], dtype=np.int64)


def _blocks(g, shapes, dtype, make):
    """Column-major tensors of the given extents inside one buffer."""
    sizes, offs, total = _packed([math.prod(s) for s in shapes])
    buf = make(g, total, dtype)
    return [buf[o:o + n].view(tuple(reversed(s))) for s, n, o in zip(shapes, sizes, offs)]


# ---- contractions ---------------------------------------------------------------------------------

def _contract_inputs(case, g):
    """Operands as stored, and the index of the view that the call takes of each (None: all of it).  With a view, the first
    operand holds all o + v orbitals along each dimension and the call takes its occupied or virtual range."""
    ext, dtype = _extents(case["ext"]), DTYPES[PRECISION_DTYPE[case["precision"]]]
    ins, views = [], []
    for n, ls in enumerate(_labels(case["expr"])[1:]):
        if n == 0 and case.get("view"):
            o, v = ext["i"], ext["a"]
            ins.append(_uniform(g, [o + v] * len(ls), dtype))
            views.append(tuple(slice(0, o) if l in "ijk" else slice(o, o + v) for l in reversed(ls)))
        else:
            ins.append(_uniform(g, [ext[l] for l in ls], dtype))
            views.append(None)
    return ins, views


def _prepare_contract(case, g):
    ext, dtype = _extents(case["ext"]), DTYPES[PRECISION_DTYPE[case["precision"]]]
    ins, _ = _contract_inputs(case, g)
    result, first = _labels(case["expr"])[:2]
    views = None
    if case.get("view"):
        o, v = ext["i"], ext["a"]
        views = [(0, d, o + v, 0 if l in "ijk" else o, 1) for d, l in enumerate(first)]
    plan = comet.Plan(case["expr"], ext, dtype, precision=case["precision"], views=views)
    out, ws = comet.colmajor_empty([ext[l] for l in result], dtype), plan.workspace()
    return {"call": lambda: plan.contract(ins, out, ws)}


def _contract_exact(expr, ops):
    """Left to right, each step a torch.einsum of two operands."""
    result, *names = _labels(expr)
    have, x = names[0], ops[0]
    for n in range(1, len(ops)):
        after = set(result).union(*names[n + 1:])
        made = [l for l in dict.fromkeys(have + names[n]) if l in after] if n + 1 < len(ops) else list(result)
        x = torch.einsum(f"{''.join(reversed(have))},{''.join(reversed(names[n]))}->{''.join(reversed(made))}", x, ops[n])
        have = tuple(made)
    return x.contiguous()


def _prepare_host(case, g):
    ext, dtype = _extents(case["ext"]), DTYPES[PRECISION_DTYPE[case["precision"]]]
    dev = _contract_inputs(case, g)[0]
    host = [torch.empty(x.shape, dtype=dtype, pin_memory=True).copy_(x) for x in dev]
    plan = comet.Plan(case["expr"], ext, dtype, precision=case["precision"])
    out = comet.colmajor_empty([ext[l] for l in _labels(case["expr"])[0]], dtype)
    host_out, ws = torch.empty(out.shape, dtype=dtype, pin_memory=True), plan.workspace()
    dev = [torch.empty_like(x) for x in dev]
    return {"call": lambda: plan.contract_host(host, host_out, dev, out, ws)}


# ---- forward and backward ---------------------------------------------------------------------------

def _chain_extents(case):
    return dict(zip("abijkl", [case["ab"], case["ab"]] + _ints(case["ijkl"])))


def _chain_inputs(case, g):
    ext = _chain_extents(case)
    result, *names = _labels(CHAIN)
    ops = [_uniform(g, [ext[l] for l in ls], torch.float32) for ls in names]
    return ops, _uniform(g, [ext[l] for l in result], torch.float32)


def _prepare_backward(case, g):
    ops, grad = _chain_inputs(case, g)
    ops = [x.requires_grad_(True) for x in ops]

    def call():
        out = autograd.einsum(CHAIN, *ops, precision=case["precision"], layout="col")
        return (out.detach(), *torch.autograd.grad(out, ops, grad))
    return {"call": call}


# ---- permutations -----------------------------------------------------------------------------------

def _copy_input(case, g):
    ext = _ints(case["ext"])
    return _uniform(g, ext, DTYPES[case["dtype"]]), ext, _ints(case["perm"])


def _prepare_copy(case, g):
    x, ext, perm = _copy_input(case, g)
    out = comet.colmajor_empty([ext[p] for p in perm], x.dtype)
    return {"call": lambda: comet.transpose(x, ext, perm, out=out)}


# ---- batched blocks ---------------------------------------------------------------------------------

def _batched_inputs(table, g):
    """Operands of every block, normal(0, 0.1)."""
    def normal(g, n, dtype):
        return torch.randn(n, generator=g, dtype=dtype, device="cuda").mul_(0.1)
    rows = table.tolist()
    return (_blocks(g, [(d, a, b, i) for a, b, c, i, j, k, d in rows], torch.float32, normal),
            _blocks(g, [(c, d, j, k) for a, b, c, i, j, k, d in rows], torch.float32, normal))


def _pointers(tensors):
    return torch.tensor([x.data_ptr() for x in tensors], dtype=torch.int64, device="cuda")


def _prepare_batched(case, g):
    table = _table(case)
    a, b = _batched_inputs(table, g)
    plan = comet.BatchedPlan(BLOCK, BLOCK_LABELS, table, torch.float32, precision=case["precision"])
    ws = plan.workspace()
    plan.prepare(ws)
    ptrs = _pointers([x for pair in zip(a, b) for x in pair])
    if case["store"]:
        _, offs, total = _packed([math.prod(r[:6]) for r in table.tolist()])
        out = torch.zeros(total, dtype=torch.float32, device="cuda")
        result, mode = torch.tensor([out.data_ptr() + 4 * o for o in offs], dtype=torch.int64, device="cuda"), 1
    else:
        out = result = torch.zeros(2 * len(table), dtype=torch.float64, device="cuda")
        mode = 0

    def call():
        plan.contract(ptrs, result, ws, mode=mode, key=1)
        return out
    return {"call": call, "keep": (a, b)}


def _mix(h):
    """MurmurHash3's 32-bit finalizer on int64 values."""
    m = 0xFFFFFFFF
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & m
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & m
    return h ^ (h >> 16)


def _hash(key, block, x):
    m = 0xFFFFFFFF
    return (_mix(key ^ _mix((block * 0x9E3779B9 + x) & m)) >> 8).double() * 2.0 ** -23 - 1.0


def _sums_exact(block, row, x, y):
    """(sum T W, sum T^2) of one block: W is a product of one factor per operand, so neither needs T itself."""
    a, b, c, i, j, k, d = row
    n = [torch.arange(e, dtype=torch.int64, device="cuda") for e in (a, b, c, i, j, k)]
    stride = np.cumprod([1, a, b, c, i, j]).tolist()
    ox = (n[3] * stride[3])[:, None, None] + (n[1] * stride[1])[:, None] + n[0] * stride[0]          # i, b, a
    oy = (n[5] * stride[5])[:, None, None] + (n[4] * stride[4])[:, None] + n[2] * stride[2]          # k, j, c
    xm = x.reshape(-1, d)                                                                            # rows (i, b, a)
    ym = y.permute(0, 1, 3, 2).reshape(-1, d)                                                        # rows (k, j, c)
    s = (_hash(1, block, ox.reshape(-1)) @ xm) @ (_hash(0xFFFFFFFE, block, oy.reshape(-1)) @ ym)
    return float(s), float(((xm.T @ xm) * (ym.T @ ym)).sum())


# ---- the triples energy -------------------------------------------------------------------------------

def _terms():
    """The base term and its images under one transposition of the virtual label on Y and of the occupied one on X."""
    out = []
    for (p, v), (q, o) in itertools.product(enumerate("cab"), enumerate("ijk")):
        x, y = [l for l in "abc" if l != v], [l for l in "ijk" if l != o]
        sign = -1.0 if (p > 0) != (q > 0) else 1.0
        out.append(f"T[a,b,c,i,j,k] = {sign} * X{len(out)}[d,{x[0]},{x[1]},{o}] * Y{len(out)}[{v},d,{y[0]},{y[1]}]")
    return out


def _triples_inputs(case, table, g):
    """Per block: the operands of every term (X, Y, X, Y, ..), uniform in [-1, 1), and the orbital energies of T's labels,
    virtual ones in [1, 2) and occupied ones in [-2, -1)."""
    def make(g, n, dtype):
        return _uniform(g, [n], dtype)
    dtype, names = DTYPES[case["dtype"]], [ls for t in _terms() for ls in _labels(t)[1:]]
    of = [dict(zip(BLOCK_LABELS, r)) for r in table.tolist()]
    ops = _blocks(g, [tuple(e[l] for l in ls) for e in of for ls in names], dtype, make)
    eps = _blocks(g, [(e[l],) for e in of for l in BLOCK_LABELS[:6]], dtype, make)
    for n, x in enumerate(eps):
        x.mul_(0.5).add_(1.5 if n % 6 < 3 else -1.5)
    return [ops[n:n + len(names)] for n in range(0, len(ops), len(names))], [eps[n:n + 6] for n in range(0, len(eps), 6)]


def _prepare_triples(case, g):
    table, dtype = _table(case), DTYPES[case["dtype"]]
    ops, eps = _triples_inputs(case, table, g)
    plan = comet.TriplesPlan(_terms(), BLOCK_LABELS, table, SIGNS, dtype)
    ws = plan.workspace()
    plan.prepare(ws)
    ops_at, eps_at = _pointers([x for o in ops for x in o]), _pointers([x for e in eps for x in e])
    energies = torch.empty(len(table), dtype=torch.float64, device="cuda")
    return {"call": lambda: plan.energy(ops_at, eps_at, energies, ws), "keep": (ops, eps)}


def _energy_exact(row, ops, eps):
    t = None
    for n, term in enumerate(_terms()):
        x = _contract_exact(re.sub(r"[-0-9.]+ \*", "", term), [ops[2 * n].double(), ops[2 * n + 1].double()])
        sign = float(re.search(r"= ([-0-9.]+)", term).group(1))
        t = x.mul_(sign) if t is None else t.add_(x, alpha=sign)
        del x
    d = torch.zeros((), dtype=torch.float64, device="cuda")
    for n, e in enumerate(eps):
        d = d + SIGNS[n] * e.double().view([-1 if 5 - n == m else 1 for m in range(6)])
    return (t.mul_(t) / d).sum()
