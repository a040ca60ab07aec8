"""The products, contractions and chains whose speed matters to a user of this library.

Every case goes through the package's public entry points on inputs shaped like the
paper's workloads: chemically sized blocks (5, 13, 23) in banded, tall-and-skinny and
windowed tensor patterns, with the block-norm filter where those chains use one.  Sizes
are those of the package's own workload generators, its tests and its benchmark.

A case is a dict: ``family`` says how the operands look, ``call`` what is done with them:

  multiply   bst.multiply: plan, allocate C, execute -- one step with fresh sparsity
  execute    plan.execute on a plan that the program keeps -- same sparsity, new values
  backward   autograd.multiply and the gradients of both operands
  sign       one Newton-Schulz step (two products, two post-filters)
  contract   bst.contract: plan, allocate the result, execute
  train      autograd.contract and the gradients of both tensors
  batch      one bst_batch_execute over many plans

A case has one block pattern; the seed gives the values.  Where a filter decides the
result's pattern, every block has the same Frobenius norm under every seed.

The exact results are formed here with torch alone: the block pairs that meet, their
products as a batch of zero-padded blocks in float64, and a sum per result block.
"""
import functools
import math

import numpy as np
import torch

from paper_1910_13555_gb300 import autograd, bst, sign

DEV = "cuda"
AO = (5, 13)                                   # block sizes of one mode of a tensor
ATOM = ((5, 13, 23), (0.4, 0.4, 0.2))          # block sizes of a matrix and their shares


def listed():
    return [
        # a few hundred products of 5 x 5 blocks: the smallest call of a chain, where the
        # plan's launches and read-backs are everything
        dict(name="plain_multiply", family="plain", call="multiply", precision="fp64", nb=40,
             size=5, occ=0.10),
        # blocks of every size from 1 to 40, both operands transposed: a basis without the
        # usual block sizes
        dict(name="ragged_multiply", family="ragged", call="multiply", precision="fp64", nm=701,
             nk=903, nn=502, smax=40, occ=0.03, ta=True, tb=True),
        # the benchmark's product: a linear-scaling step, filtered, fresh sparsity each time
        dict(name="banded_multiply", family="banded", call="multiply", precision="fp64", nb=4000,
             occ=0.01),
        # the same product repeated on a kept plan in emulated FP64
        dict(name="banded_emulated", family="banded", call="execute", precision="emu_bf16",
             nb=4000, occ=0.01),
        # single-precision accuracy (preconditioners, early iterations) on a kept plan
        dict(name="banded_tf32x3", family="banded", call="execute", precision="tf32x3", nb=2000,
             occ=0.02),
        # forward and both gradients of a banded product
        dict(name="banded_backward", family="banded", call="backward", precision="fp64", nb=2000,
             occ=0.02),
        # one step of the matrix-sign iteration: chained filtered products and post-filters
        dict(name="sign_step", family="sign", call="sign", precision="fp64", nb=2000, width=12),
        # C = A^T B with a long inner dimension and a small C, the split left to the library
        dict(name="tall_skinny", family="tall_skinny", call="multiply", precision="fp64",
             nk=100000, nmn=400),
        # a tall A times a small B, added to an existing C with alpha and beta
        dict(name="small_b_accumulate", family="small_b", call="multiply", precision="fp64",
             nm=20000, nk=400),
        # a rank-3 contraction over two index pairs and its gradients
        dict(name="rank3_train", family="rank3", call="train", precision="fp64", nP=500, nao=1000),
        # a rank-4 with a rank-3 tensor: permuted operand, permuted result
        dict(name="rank4_contract", family="rank4", call="contract", precision="fp64", nP=400,
             nao=400),
        # many independent products of very different sizes in one launch
        dict(name="batch", family="batched", call="batch", precision="fp64", nprob=32, nmin=100,
             nmax=800),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges."""
    family = rng.choice(["plain", "ragged", "banded", "banded", "banded", "sign", "tall_skinny",
                         "small_b", "rank3", "rank4", "batched"])
    if family == "plain":
        nb = int(_log(rng, 24, 400))
        return dict(family=family, call=rng.choice(["multiply", "execute"]),
                    precision=rng.choice(["fp64", "emu_bf16", "tf32x3"]), nb=nb,
                    size=rng.choice([1, 2, 4, 5, 7, 13, 16, 23]), occ=_log(rng, 0.05, 0.2))
    if family == "ragged":
        return dict(family=family, call=rng.choice(["multiply", "execute", "backward"]),
                    precision="fp64", nm=int(_log(rng, 80, 900)), nk=int(_log(rng, 80, 900)),
                    nn=int(_log(rng, 80, 900)), smax=rng.choice([3, 9, 17, 33, 40]),
                    occ=_log(rng, 0.02, 0.04), ta=rng.random() < 0.5, tb=rng.random() < 0.5)
    if family == "banded":
        nb = int(_log(rng, 60, 4000))
        call = rng.choice(["multiply", "execute", "backward"])
        prec = rng.choice(["fp64", "emu_bf16", "tf32x3"]) if call == "execute" else "fp64"
        most = min(0.2, 0.01 * (4000 / nb) ** 1.5) * (1.0 if call != "backward" else 0.6)
        return dict(family=family, call=call, precision=prec, nb=nb, occ=_log(rng, 0.004, most))
    if family == "sign":
        return dict(family=family, call="sign", precision="fp64", nb=int(_log(rng, 50, 2000)),
                    width=rng.randint(2, 12))
    if family == "tall_skinny":
        return dict(family=family, call=rng.choice(["multiply", "execute"]),
                    precision=rng.choice(["fp64", "fp64", "emu_bf16"]),
                    nk=int(_log(rng, 1000, 100000)), nmn=int(_log(rng, 70, 400)))
    if family == "small_b":
        return dict(family=family, call=rng.choice(["multiply", "execute"]), precision="fp64",
                    nm=int(_log(rng, 300, 20000)), nk=int(_log(rng, 70, 400)))
    if family == "rank3":
        return dict(family=family, call=rng.choice(["contract", "train"]), precision="fp64",
                    nP=int(_log(rng, 20, 500)), nao=int(_log(rng, 60, 1000)))
    if family == "rank4":
        return dict(family=family, call=rng.choice(["contract", "train"]), precision="fp64",
                    nP=int(_log(rng, 20, 200)), nao=int(_log(rng, 40, 400)))
    return dict(family=family, call="batch", precision=rng.choice(["fp64", "emu_bf16"]),
                nprob=rng.randint(4, 32), nmin=int(_log(rng, 30, 100)),
                nmax=int(_log(rng, 200, 700)))


# ---- inputs -----------------------------------------------------------------------------


class _Blocks:
    """Packed blocks in canonical order: per-mode sizes (numpy), index (CUDA int64 [n, rank])
    and data (CUDA float64)."""

    def __init__(self, sizes, index, data=None):
        self.sizes, self.index, self.data = sizes, index, data

    @functools.cached_property
    def shapes(self):
        return torch.stack([_dev(s)[self.index[:, d]] for d, s in enumerate(self.sizes)], 1)

    @property
    def lens(self):
        return self.shapes.prod(1)

    @property
    def nelem(self):
        return int(self.lens.sum()) if len(self.index) else 0


def _dev(a):
    return torch.as_tensor(np.asarray(a, np.int64)).to(DEV)


PATTERN = 1002                                 # seeds the block sizes and patterns


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _fill(b, g, dist="uniform", norm=None):
    """Values from the generator g; each block scaled to its Frobenius norm, if given."""
    n = b.nelem
    if dist == "normal":
        b.data = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    else:
        b.data = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2 - 1
    if norm is not None:
        b.data *= torch.repeat_interleave(norm / _norms(b), b.lens)
    return b


def _spread(g, n):
    """Block norms scatter by a factor around their trend."""
    return torch.exp(0.2 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))


def _ordered(grid, *modes):
    """Index of the given tuples in lexicographic order, each once."""
    key = modes[0].clone()
    for n, m in zip(grid[1:], modes[1:]):
        key = key * n + m
    key = torch.unique(key)
    out = []
    for n in reversed(grid[1:]):
        out.append(key % n)
        key = key // n
    return torch.stack([key] + out[::-1], 1)


def _bernoulli(g, nr, nc, p):
    return (torch.rand(nr, nc, generator=g, device=DEV) < p).nonzero()


def _atom_sizes(r, n):
    return r.choice(np.array(ATOM[0], np.int32), n, p=np.array(ATOM[1])).astype(np.int32)


def _window(g, centre, n, window, p, lists=2):
    """Rows r and, for each of `lists` modes, columns (centre_r + offset) mod n of the
    offsets in [0, window) kept with probability p."""
    keep = torch.rand(len(centre), *[min(window, n)] * lists, generator=g, device=DEV) < p
    at = keep.nonzero()
    c = centre[at[:, 0]]
    return at[:, 0], [(c + at[:, 1 + q]) % n for q in range(lists)]


class _Product:
    """C = alpha op(A) op(B) + beta C_in with the filter eps."""

    def __init__(self, A, B, Cin=None, alpha=1.0, beta=0.0, eps=0.0, ta=False, tb=False):
        self.A, self.B, self.Cin = A, B, Cin
        self.alpha, self.beta, self.eps, self.ta, self.tb = alpha, beta, eps, ta, tb


def _product(c, seed):
    g, r, v = _gen(PATTERN), np.random.default_rng(PATTERN), _gen(seed)
    f = c["family"]
    if f == "plain":
        s = np.full(c["nb"], c["size"], np.int32)
        return _Product(*[_fill(_Blocks([s, s], _bernoulli(g, c["nb"], c["nb"], c["occ"])), v)
                          for _ in range(2)])
    if f == "ragged":
        sm, sk, sn = (r.integers(1, c["smax"] + 1, c[k]).astype(np.int32)
                      for k in ("nm", "nk", "nn"))
        a, b = ([sk, sm] if c["ta"] else [sm, sk]), ([sn, sk] if c["tb"] else [sk, sn])
        return _Product(*[_fill(_Blocks(s, _bernoulli(g, len(s[0]), len(s[1]), c["occ"])), v)
                          for s in (a, b)], ta=c["ta"], tb=c["tb"])
    if f == "banded":
        # kept with probability ~ exp(-|i - j| / 200), mean occupancy occ; entries fall off
        # as exp(-|i - j| / 50)
        s = _atom_sizes(r, c["nb"])
        d = torch.arange(c["nb"], device=DEV)
        p = torch.exp(-(d[:, None] - d[None, :]).abs().float() / 200.0)
        p *= c["occ"] / float(p.mean())
        ops = []
        for _ in range(2):
            b = _Blocks([s, s], _bernoulli(g, c["nb"], c["nb"], p))
            far = (b.index[:, 0] - b.index[:, 1]).abs().double()
            norm = torch.exp(-far / 50.0) * b.lens.sqrt() * _spread(g, len(far))
            ops.append(_fill(b, v, "normal", norm))
        return _Product(*ops, eps=1e-8)
    if f == "tall_skinny":
        # row block r keeps columns of the window of 60 that starts at its centre, 1 in 30
        sk = r.integers(20, 51, c["nk"]).astype(np.int32)
        sm = r.choice(np.array(AO, np.int32), c["nmn"]).astype(np.int32)
        centre = _dev(r.integers(0, c["nmn"], c["nk"]))
        ops = []
        for _ in range(2):
            rows, (cols,) = _window(g, centre, c["nmn"], 60, 1 / 30, 1)
            ops.append(_fill(_Blocks([sk, sm], _ordered([c["nk"], c["nmn"]], rows, cols)), v))
        return _Product(*ops, ta=True)
    if f == "small_b":
        sm = r.integers(20, 51, c["nm"]).astype(np.int32)
        sk = r.choice(np.array(AO, np.int32), c["nk"]).astype(np.int32)
        centre = _dev(r.integers(0, c["nk"], c["nm"]))
        rows, (cols,) = _window(g, centre, c["nk"], 60, 1 / 30, 1)
        A = _fill(_Blocks([sm, sk], _ordered([c["nm"], c["nk"]], rows, cols)), v)
        at = torch.arange(c["nk"], device=DEV)
        rows, (cols,) = _window(g, at, c["nk"], 20, 0.5, 1)
        B = _fill(_Blocks([sk, sk], _ordered([c["nk"], c["nk"]], rows, cols)), v)
        rows, (cols,) = _window(g, centre, c["nk"], 60, 1 / 6, 1)
        Ci = _fill(_Blocks([sm, sk], _ordered([c["nm"], c["nk"]], rows, cols)), v)
        return _Product(A, B, Ci, alpha=-0.5, beta=1.5)
    raise ValueError(f)


def _batch_products(c, seed):
    out = []
    for q in range(c["nprob"]):
        r = np.random.default_rng((PATTERN, q))
        g, v = _gen(int(r.integers(1 << 40))), _gen(seed * 1000 + q)
        # sizes and occupancies over the whole range, the largest product bounded
        n = int(math.exp(r.uniform(math.log(c["nmin"]), math.log(c["nmax"]))))
        occ = math.exp(r.uniform(math.log(1e-3), math.log(1e-1)))
        s = _atom_sizes(r, n)
        ops = []
        for _ in range(2):
            b = _Blocks([s, s], _bernoulli(g, n, n, occ))
            far = torch.rand(len(b.index), generator=g, device=DEV, dtype=torch.float64)
            ops.append(_fill(b, v, "uniform", 10.0 ** (-8 * far) * (b.lens / 3.0).sqrt()))
        out.append(_Product(*ops, eps=1e-10))
    return out


def _sign_input(c, seed):
    """A symmetric matrix with eigenvalues away from 0 near its diagonal blocks, weakly coupled
    to the neighbours within `width` blocks, scaled into [-1, 1] by its largest row sum, in a
    basis of each block that the seed rotates (which leaves all block norms of the chain)."""
    g, r, v = _gen(PATTERN), np.random.default_rng(PATTERN), _gen(seed)
    nb = c["nb"]
    s = _atom_sizes(r, nb)
    sd = _dev(s)
    mx = max(ATOM[0])
    inside = torch.arange(mx, device=DEV)[None, :] < sd[:, None]

    def rotations(g):
        x = torch.randn(nb, mx, mx, generator=g, device=DEV, dtype=torch.float64)
        x = x * (inside[:, :, None] & inside[:, None, :])
        return torch.linalg.qr(x + torch.diag_embed((~inside).double()))[0]

    q = rotations(g)
    lam = 0.3 + 0.7 * torch.rand(nb, mx, generator=g, device=DEV, dtype=torch.float64)
    lam *= torch.where(torch.rand(nb, mx, generator=g, device=DEV) < 0.5, -1.0, 1.0)
    diag = (q * lam[:, None, :]) @ q.transpose(1, 2)
    keep = torch.rand(nb, c["width"], generator=g, device=DEV) < 0.5
    at = keep.nonzero()
    i, j = at[:, 0], at[:, 0] + 1 + at[:, 1]
    i, j = i[j < nb], j[j < nb]
    off = torch.randn(len(i), mx, mx, generator=g, device=DEV, dtype=torch.float64)
    off *= (0.1 / torch.sqrt((sd[i] * sd[j]).double()))[:, None, None]
    d = torch.arange(nb, device=DEV)
    idx = torch.cat([torch.stack([d, d], 1), torch.stack([i, j], 1), torch.stack([j, i], 1)])
    blk = torch.cat([diag, off, off.transpose(1, 2)])
    order = torch.argsort(idx[:, 0] * nb + idx[:, 1])
    b = _Blocks([s, s], idx[order])
    b.data = _unpad(blk[order], b.shapes)
    p = _pad(b.data, b.shapes)
    rows = torch.zeros(nb, p.shape[1], dtype=torch.float64, device=DEV)
    rows.index_add_(0, b.index[:, 0], p.abs().sum(2))
    q = rotations(v)
    p = q[b.index[:, 0]] @ (p / rows.max()) @ q[b.index[:, 1]].transpose(1, 2)
    b.data = _unpad(p, b.shapes)
    return b


def _tensors(c, seed):
    g, r, v = _gen(PATTERN), np.random.default_rng(PATTERN), _gen(seed)
    sp = np.full(c["nP"], 30, np.int32)
    sa = r.choice(np.array(AO, np.int32), c["nao"]).astype(np.int32)
    centre = _dev(r.integers(0, c["nao"], c["nP"]))
    nP, n = c["nP"], c["nao"]

    def tensor(window, p, modes):
        P, m = _window(g, centre, n, window, p, modes)
        return _fill(_Blocks([sp] + [sa] * modes, _ordered([nP] + [n] * modes, P, *m)), v)

    if c["family"] == "rank3":
        return tensor(20, 0.25, 2), tensor(20, 0.25, 2)
    return tensor(8, 0.04, 3), tensor(8, 0.25, 2)


#: contracted and free modes, result order; the letters of the padded blocks
_CON = {
    "rank3": dict(c1=[0, 2], c2=[0, 1], f1=[1], f2=[2], order=None, t="pmv", u="pvl", r="ml"),
    "rank4": dict(c1=[0, 2], c2=[0, 1], f1=[1, 3], f2=[2], order=[0, 2, 1], t="pmvl", u="pvs",
                  r="msl"),
}


# ---- what a program holds, and one pass ---------------------------------------------------


def _matrix(b):
    i = b.index.cpu().numpy()
    h = bst.bst_matrix_create(bst.context(), b.sizes[0], b.sizes[1], i[:, 0], i[:, 1], b.data)
    return bst.Matrix(h, b.data)


def _tensor(b):
    h = bst.bst_tensor_create(bst.context(), b.sizes, b.index.cpu().numpy(), b.data)
    return bst.Tensor(h, b.data)


class _Held:
    """What a program keeps between passes."""

    def __init__(self, **kw):
        self.batch = None
        self.__dict__.update(kw)

    def __del__(self):
        if self.batch is not None:
            bst.bst_batch_destroy(self.batch)


def _plan(p, A, B, Ci):
    plan = bst.multiply_plan(A, B, Ci, p.eps, "T" if p.ta else "N", "T" if p.tb else "N")
    plan.alloc_result()
    return plan


def prepare(case, seed):
    call = case["call"]
    if call == "sign":
        return _Held(case=case, X=_matrix(_sign_input(case, seed)))
    if call in ("contract", "train"):
        T, U = (_tensor(b) for b in _tensors(case, seed))
        if call == "train":
            T.data.requires_grad_(True)
            U.data.requires_grad_(True)
        return _Held(case=case, T=T, U=U)
    if call == "batch":
        plans = [_plan(p, _matrix(p.A), _matrix(p.B), None) for p in _batch_products(case, seed)]
        torch.cuda.synchronize()
        return _Held(case=case, plans=plans, one=np.ones(len(plans)), zero=np.zeros(len(plans)),
                     batch=bst.bst_batch_create(bst.context(), [q.handle for q in plans]))
    p = _product(case, seed)
    A, B, Ci = _matrix(p.A), _matrix(p.B), None if p.Cin is None else _matrix(p.Cin)
    st = _Held(case=case, A=A, B=B, Ci=Ci, alpha=p.alpha, beta=p.beta, eps=p.eps,
               ta="T" if p.ta else "N", tb="T" if p.tb else "N")
    if call == "backward":
        A.data.requires_grad_(True)
        B.data.requires_grad_(True)
    if call == "execute":
        st.plan = _plan(p, A, B, Ci)
        if case["precision"] != "fp64":
            # a plan that is kept for many products has its tensor-core schedule, which the
            # library builds with the second execute
            for _ in range(2):
                st.plan.execute(p.alpha, p.beta, case["precision"])
    return st


def run(st):
    c = st.case
    call, prec = c["call"], bst.PRECISIONS[c["precision"]]
    if call == "execute":
        st.plan.execute(st.alpha, st.beta, prec, split_k=0 if c["family"] == "tall_skinny" else 1)
        return st.plan.result.data
    if call == "multiply":
        p = bst.multiply(st.A, st.B, st.Ci, st.alpha, st.beta, st.eps, st.ta, st.tb, prec,
                         split_k=0 if c["family"] == "tall_skinny" else 1)
        return p.result.data
    if call == "backward":
        y, _ = autograd.multiply(st.A, st.B, None, st.alpha, 0.0, st.eps, st.ta, st.tb, prec)
        da, db = torch.autograd.grad(y, (st.A.data, st.B.data), y.detach())
        return [y.detach(), da, db]
    if call == "sign":
        x, _ = sign.sign_step(st.X, 1e-8, 1e-7, prec)
        return x.data
    if call == "batch":
        bst.bst_batch_execute(st.batch, st.one, st.zero, prec)
        return [p.result.data for p in st.plans]
    k = _CON[c["family"]]
    if call == "contract":
        p = bst.contract(st.T, st.U, k["c1"], k["c2"], k["f1"], k["f2"], k["order"],
                         precision=prec)
        return p.result.data
    y, _ = autograd.contract(st.T, st.U, k["c1"], k["c2"], k["f1"], k["f2"], k["order"],
                             precision=prec)
    dt, du = torch.autograd.grad(y, (st.T.data, st.U.data), y.detach())
    return [y.detach(), dt, du]


# ---- the exact results, with torch alone ----------------------------------------------------


def _mask(shapes, most):
    m = torch.ones((len(shapes),) + tuple(most), dtype=torch.bool, device=DEV)
    for d, k in enumerate(most):
        view = [len(shapes)] + [1] * len(most)
        view[1 + d] = k
        m &= (torch.arange(k, device=DEV)[None, :] < shapes[:, d:d + 1]).view(view)
    return m


def _chunks(n, per):
    step = max(1, int(2e8 // max(per, 1)))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _most(shapes):
    return [int(v) for v in shapes.max(0).values] if len(shapes) else [1] * shapes.shape[1]


def _pad(data, shapes, most=None):
    most = most or _most(shapes)
    out = torch.zeros((len(shapes),) + tuple(most), dtype=torch.float64, device=DEV)
    at = 0
    for a, b in _chunks(len(shapes), math.prod(most)):
        m = _mask(shapes[a:b], most)
        n = int(m.sum())
        out[a:b].masked_scatter_(m, data[at:at + n])
        at += n
    return out


def _unpad(p, shapes):
    out = []
    for a, b in _chunks(len(shapes), math.prod(p.shape[1:])):
        out.append(torch.masked_select(p[a:b], _mask(shapes[a:b], p.shape[1:])))
    return torch.cat(out) if out else torch.zeros(0, dtype=torch.float64, device=DEV)


def _meet(ka, kb):
    """All (a, b) with ka[a] == kb[b]."""
    order = torch.argsort(kb, stable=True)
    kb = kb[order]
    lo = torch.searchsorted(kb, ka)
    cnt = torch.searchsorted(kb, ka, right=True) - lo
    a = torch.repeat_interleave(torch.arange(len(ka), device=DEV), cnt)
    start = torch.cumsum(cnt, 0) - cnt
    return a, order[lo[a] + torch.arange(len(a), device=DEV) - start[a]]


def _norms(b):
    return torch.segment_reduce(b.data * b.data, "sum", lengths=b.lens).sqrt()


def _pairs(p):
    """The kept block pairs, C's index and each pair's C block (and C_in's)."""
    ai, ak = (p.A.index[:, 1], p.A.index[:, 0]) if p.ta else (p.A.index[:, 0], p.A.index[:, 1])
    bk, bj = (p.B.index[:, 1], p.B.index[:, 0]) if p.tb else (p.B.index[:, 0], p.B.index[:, 1])
    a, b = _meet(ak, bk)
    if p.eps > 0:
        keep = _norms(p.A)[a] * _norms(p.B)[b] >= p.eps
        a, b = a[keep], b[keep]
    sr, sc = p.A.sizes[1 if p.ta else 0], p.B.sizes[0 if p.tb else 1]
    n = len(sc)
    key = ai[a] * n + bj[b]
    if p.Cin is not None:
        key = torch.cat([key, p.Cin.index[:, 0] * n + p.Cin.index[:, 1]])
    u, inv = torch.unique(key, return_inverse=True)
    C = _Blocks([sr, sc], torch.stack([u // n, u % n], 1))
    return a, b, inv[:len(a)], inv[len(a):], C


def _sum(eq, X, Y, x, y, into, n, shape):
    """sum over the pairs of einsum(eq, X[x], Y[y]) into n padded blocks."""
    out = torch.zeros((n,) + tuple(shape), dtype=torch.float64, device=DEV)
    per = max(math.prod(X.shape[1:]), math.prod(Y.shape[1:]), math.prod(shape))
    for a, b in _chunks(len(x), per):
        out.index_add_(0, into[a:b], torch.einsum(eq, X[x[a:b]], Y[y[a:b]]))
    return out


def _multiply(p, back=False):
    a, b, c, ci, C = _pairs(p)
    A, B = _pad(p.A.data, p.A.shapes), _pad(p.B.data, p.B.shapes)
    ea, eb = "nkm" if p.ta else "nmk", "njk" if p.tb else "nkj"
    m, j = A.shape[2 if p.ta else 1], B.shape[1 if p.tb else 2]
    out = _sum(f"{ea},{eb}->nmj", A, B, a, b, c, len(C.index), (m, j)).mul_(p.alpha)
    if p.Cin is not None:
        P = _pad(p.Cin.data, p.Cin.shapes, (m, j))
        out.index_add_(0, ci, P, alpha=p.beta)
    C.data = _unpad(out, C.shapes)
    if not back:
        return C
    da = _sum(f"nmj,{eb}->{ea}", out, B, c, b, a, len(A), A.shape[1:]).mul_(p.alpha)
    db = _sum(f"{ea},nmj->{eb}", A, out, a, c, b, len(B), B.shape[1:]).mul_(p.alpha)
    return C, _unpad(da, p.A.shapes), _unpad(db, p.B.shapes)


def _filter(b, eps):
    keep = _norms(b) >= eps
    out = _Blocks(b.sizes, b.index[keep])
    out.data = b.data[torch.repeat_interleave(keep, b.lens)]
    return out


def _contraction_pairs(c, T, U):
    n, fam = c["nao"], c["family"]
    t, u = _meet(T.index[:, 0] * n + T.index[:, 2], U.index[:, 0] * n + U.index[:, 1])
    sa = T.sizes[1]
    if fam == "rank3":
        modes = [T.index[t, 1], U.index[u, 2]]
    else:
        modes = [T.index[t, 1], U.index[u, 2], T.index[t, 3]]
    key = modes[0]
    for m in modes[1:]:
        key = key * n + m
    uniq, inv = torch.unique(key, return_inverse=True)
    idx, k = [], uniq
    for _ in modes[1:]:
        idx.append(k % n)
        k = k // n
    return t, u, inv, _Blocks([sa] * len(modes), torch.stack([k] + idx[::-1], 1))


def _contract(c, T, U, back):
    k = _CON[c["family"]]
    t, u, r, R = _contraction_pairs(c, T, U)
    X, Y = _pad(T.data, T.shapes), _pad(U.data, U.shapes)
    shape = [max(AO)] * len(k["r"])
    et, eu, er = "n" + k["t"], "n" + k["u"], "n" + k["r"]
    out = _sum(f"{et},{eu}->{er}", X, Y, t, u, r, len(R.index), shape)
    R.data = _unpad(out, R.shapes)
    if not back:
        return R.data
    dt = _sum(f"{er},{eu}->{et}", out, Y, r, u, t, len(X), X.shape[1:])
    du = _sum(f"{et},{er}->{eu}", X, out, t, r, u, len(Y), Y.shape[1:])
    return [R.data, _unpad(dt, T.shapes), _unpad(du, U.shapes)]


def exact(case, seed):
    call = case["call"]
    if call == "sign":
        X = _sign_input(case, seed)
        T = _filter(_multiply(_Product(X, X, eps=1e-8)), 1e-7)
        return _filter(_multiply(_Product(T, X, X, -0.5, 1.5, 1e-8)), 1e-7).data
    if call == "batch":
        return [_multiply(p).data for p in _batch_products(case, seed)]
    if call in ("contract", "train"):
        return _contract(case, *_tensors(case, seed), call == "train")
    p = _product(case, seed)
    if call == "backward":
        C, da, db = _multiply(p, True)
        return [C.data, da, db]
    return _multiply(p).data


# ---- the work of one pass -----------------------------------------------------------------


def _product_work(p):
    """Operand blocks that some kept product uses are read once, C (and C_in) once."""
    a, b, _, _, C = _pairs(p)
    sa, sb = p.A.shapes, p.B.shapes
    flops = 2.0 * float((sa[a].prod(1) * sb[b, 0 if p.tb else 1]).sum())
    read = sum(int(x.lens[torch.unique(i)].sum()) for x, i in ((p.A, a), (p.B, b)))
    read += p.Cin.nelem if p.Cin is not None and p.beta else 0
    return 8.0 * read, 8.0 * C.nelem, flops


def work(case):
    call = case["call"]
    if call == "sign":
        X = _sign_input(case, 0)
        T = _filter(_multiply(_Product(X, X, eps=1e-8)), 1e-7)
        p = _Product(T, X, X, -0.5, 1.5, 1e-8)
        Y = _filter(_multiply(p), 1e-7)
        _, _, f1 = _product_work(_Product(X, X, eps=1e-8))
        _, _, f2 = _product_work(p)
        return {"bytes": 8.0 * (X.nelem + Y.nelem), "flops": f1 + f2}
    if call == "batch":
        w = [_product_work(p) for p in _batch_products(case, 0)]
        return {"bytes": sum(r + o for r, o, _ in w), "flops": sum(f for _, _, f in w)}
    if call in ("contract", "train"):
        T, U = _tensors(case, 0)
        t, u, _, R = _contraction_pairs(case, T, U)
        flops = 2.0 * float((T.shapes[t].prod(1) * U.shapes[u, 2]).sum())
        nbytes = 8.0 * (T.nelem + U.nelem + R.nelem)
        if call == "train":
            return {"bytes": nbytes + 8.0 * (T.nelem + U.nelem), "flops": 3 * flops}
        return {"bytes": nbytes, "flops": flops}
    r, o, flops = _product_work(_product(case, 0))
    if call == "backward":
        return {"bytes": 2 * r + o, "flops": 3 * flops}
    return {"bytes": r + o, "flops": flops}
