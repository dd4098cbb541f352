"""Timed cases of the library: what users have it do, through its public calls.

A case is a dict of plain values; `op` names the call:

  product   z = op(a) op(b) on matrix fields with `links` links per site, or
            matrix times vector (`form` av), in each storage format
  tree      a fused expression, compiled (commutator, sum, nested) or
            interpreted (factored, adjproduct)
  batch     z = a b + c d on `count` lattices of mixed sizes, one graph launch
  autograd  forward and backward of a tree through torch.autograd
  dslash    the Wilson hopping term
  solver    q = p - kappa D p and <p, q>: one operator application of an
            iterative solver
  hop       the colour hopping term on a vector or a matrix field
  io        a gauge configuration is taken in (pack), projected to SU(3) and
            given out again (unpack)

Outputs come back in the fields' own order, [link][component][site][re, im]
(site-blocked layouts: one array of the whole blocks and one of the rest), so
that pad sites are left out and nothing is copied.
"""
import numpy as np
import torch

import paper_1710_09409_gb300 as su3s

PREC = {"f64": su3s.F64, "f32": su3s.F32, "bf16": su3s.BF16, "f16": su3s.F16,
        "f64_c12": su3s.F64_C12, "f32_c12": su3s.F32_C12}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16,
         "f64_c12": torch.float64, "f32_c12": torch.float32}
REAL_BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2, "f64_c12": 8, "f32_c12": 4}
MATH = {"default": su3s.MATH_DEFAULT, "f64": su3s.MATH_F64, "fx": su3s.MATH_FX}
KAPPA = 0.124
BATCH_SHAPES = ((4, 4, 4, 4), (8, 8, 8, 8), (12, 12, 12, 12), (16, 16, 16, 32), (24, 24, 24, 24))

# matrices read by each tree, flops per site (complex multiply 6, add 2)
TREES = {"commutator": ("ab", 414), "sum": ("abcd", 414), "nested": ("abcd", 432),
         "factored": ("abcd", 234), "adjproduct": ("abc", 396)}


# ------------------------------------------------------------------- cases
def _case(name, op, dims, **kw):
    c = {"op": op, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3]}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # one product on the smallest lattice of the tests and the sweep: latency and host path
        _case("product_8", "product", (8, 8, 8, 8), links=1, form="ab", storage="f64",
              layout="soa", math="default"),
        # the Lorentz-indexed product z_mu = a_mu b_mu of two link fields: bulk streaming
        _case("links_product_32", "product", (32, 32, 32, 32), links=4, form="ab", storage="f64",
              layout="soa", math="default"),
        # reduced storage on a lattice whose extents divide nothing
        _case("product_bf16_ragged", "product", (45, 47, 46, 49), links=1, form="ab",
              storage="bf16", layout="soa", math="default"),
        # adj(a) b - b adj(a): the densest fused tree of the catalogue
        _case("commutator_40", "tree", (40, 40, 40, 40), tree="commutator", layout="soa",
              math="default"),
        # (a b) c + 0.5 d in the accuracy-first arithmetic on the site-blocked layout
        _case("nested_fx_blocked_32", "tree", (32, 32, 32, 32), tree="nested", layout="aosoa64",
              math="fx"),
        # many small lattices of uneven volumes, one launch
        _case("batch_64", "batch", (4, 4, 4, 4), count=64),
        # training direction: forward and backward of a b + c d through torch.autograd
        _case("autograd_32", "autograd", (32, 32, 32, 32), tree="sum"),
        # the Wilson operator on a production-shaped lattice
        _case("dslash_32x64", "dslash", (32, 32, 32, 64), layout="soa", math="default"),
        # one solver iteration's operator and inner product on a small lattice
        _case("solver_16x32", "solver", (16, 16, 16, 32)),
        # the colour hopping term on vectors, odd extents
        _case("hop_vector_ragged", "hop", (47, 45, 46, 49), kind="vector", layout="soa",
              math="default"),
        # a tree outside the compiled catalogue, a (b + c) - d, odd extents
        _case("interpreted_ragged", "tree", (31, 33, 32, 35), tree="factored", layout="soa",
              math="default"),
        # configuration in, projection, configuration out, odd extents
        _case("gauge_io_ragged", "io", (23, 25, 24, 47), storage="f64"),
    ]


def _extents(rng, lo, hi):
    """Four extents whose volume is log-uniform in lo..hi, half of them with odd ones among them."""
    v = float(np.exp(rng.uniform(np.log(lo), np.log(hi))))
    base = v ** 0.25
    d = [max(2, int(round(base * rng.uniform(0.75, 1.3)))) for _ in range(3)]
    d.append(max(2, int(round(v / (d[0] * d[1] * d[2])))))
    if rng.random() < 0.5:
        d = [e + (e & 1) for e in d]
    while d[0] * d[1] * d[2] * d[3] > hi:
        d[d.index(max(d))] -= 1
    return tuple(d)


def draw(rng):
    op = rng.choice(["product", "product", "tree", "tree", "batch", "autograd", "dslash",
                     "solver", "hop", "io"])
    layout = rng.choice(["soa", "soa", "aosoa32", "aosoa64"])
    math = rng.choice(["default", "default", "default", "fx"])
    if op == "product":
        storage = rng.choice(["f64", "f64", "f32", "bf16", "f16", "f64_c12", "f32_c12"])
        form = rng.choice(["ab", "adj(a)b", "a adj(b)"] + (["av"] if "c12" not in storage else []))
        if storage != "f64":
            math = "default"
        links = rng.choice([1, 1, 4]) if form == "ab" else 1
        return _case(None, op, _extents(rng, 1500, 3.5e6 / links), links=links, form=form,
                     storage=storage, layout=layout, math=math)
    if op == "tree":
        return _case(None, op, _extents(rng, 4000, 3e6), tree=rng.choice(sorted(TREES)),
                     layout=layout, math=math)
    if op == "batch":
        d = _extents(rng, 200, 2e4)
        return _case(None, op, d, count=rng.randint(8, 64))
    if op == "autograd":
        return _case(None, op, _extents(rng, 4000, 1.2e6), tree=rng.choice(["product", "sum", "nested"]))
    if op == "dslash":
        return _case(None, op, _extents(rng, 4000, 2.2e6), layout=layout, math=math)
    if op == "solver":
        return _case(None, op, _extents(rng, 4000, 1.2e6))
    if op == "hop":
        kind = rng.choice(["vector", "vector", "matrix"])
        return _case(None, op, _extents(rng, 4000, 1.2e6 if kind == "matrix" else 4.8e6), kind=kind,
                     layout=layout, math=math)
    return _case(None, op, _extents(rng, 2000, 6.5e5), storage="f64")


def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _batch_dims(case):
    """Lattices of a batch: the mixed volumes in turn, the case's own lattice as one of them."""
    shapes = [_dims(case)] + list(BATCH_SHAPES[1:])
    return [shapes[i % len(shapes)] for i in range(case["count"])]


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gauss(g, n, *tail):
    return torch.randn((n,) + tail, dtype=torch.float64, device="cuda", generator=g)


def _su3(g, n):
    """n SU(3) matrices as (n, 3, 3) complex: Gaussian rows, Gram-Schmidt, determinant phase removed."""
    m = torch.view_as_complex(_gauss(g, n, 3, 3, 2))
    r0 = m[:, 0] / m[:, 0].abs().square().sum(1, keepdim=True).sqrt()
    r1 = m[:, 1]
    for _ in range(2):
        r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(1, keepdim=True).sqrt()
    return torch.stack((r0, r1, torch.linalg.cross(r0, r1).conj()), 1)


def _canonical(z):
    return torch.view_as_real(z.resolve_conj().contiguous())


def _stored(canon, storage):
    """The values that the storage format holds (what a user of reduced storage starts from)."""
    return canon.to(DTYPE[storage]).double()


def _layout(name):
    return (su3s.SOA, 64) if name == "soa" else (su3s.AOSOA, int(name[5:]))


def _field(lat, canon, kind=su3s.MATRIX, links=1, storage="f64", layout="soa"):
    lay, block = _layout(layout)
    f = su3s.Field(lat, kind, links, PREC[storage], lay, block)
    f.pack(canon.contiguous())
    return f


def _inputs(case, seed):
    """Canonical float64 inputs of a case, in the order they are drawn."""
    g = _generator(seed)
    v, op = _volume(case), case["op"]
    if op == "product":
        n = v * case["links"]
        second = _gauss(g, n, 3, 2) if case["form"] == "av" else _canonical(_su3(g, n))
        return [_stored(_canonical(_su3(g, n)), case["storage"]), _stored(second, case["storage"])]
    if op == "tree":
        return [_canonical(_su3(g, v)) for _ in TREES[case["tree"]][0]]
    if op == "batch":
        n = sum(d[0] * d[1] * d[2] * d[3] for d in _batch_dims(case))
        return [_canonical(_su3(g, n)) for _ in range(4)]
    if op == "autograd":
        names = "ab" if case["tree"] == "product" else "abcd"
        return [_canonical(_su3(g, v)) for _ in names] + [_gauss(g, v, 3, 3, 2)]
    if op in ("dslash", "solver"):
        return [_canonical(_su3(g, 4 * v)), _gauss(g, 4 * v, 3, 2)]
    if op == "hop":
        return [_canonical(_su3(g, 4 * v)),
                _gauss(g, v, 3, 2) if case["kind"] == "vector" else _canonical(_su3(g, v))]
    # a configuration as files hold it: single-precision entries, unitary to their rounding
    return [_canonical(_su3(g, 4 * v)).float().double()]


# ----------------------------------------------------------------- outputs
def _views(f):
    """The field's values without pad sites, as views of its tensor."""
    width = {su3s.MATRIX: 9, su3s.VECTOR: 3}[f.kind]
    if f.prec in (su3s.F64_C12, su3s.F32_C12):
        width = 6
    t = f.tensor if f.prec == su3s.F64 else f.tensor.view(f.stored_dtype)
    v = f.lattice.volume
    if f.layout == su3s.SOA:
        return t.view(f.nmu, width, -1, 2)[:, :, :v]
    t = t.view(-1, f.nmu, width, f.block, 2)
    whole, rest = divmod(v, f.block)
    return [t[:whole], t[whole:whole + 1, :, :, :rest]] if rest else [t]


def _laid_out(z, case, links=1, layout="soa"):
    """(V * links, ...) complex values in the order of _views."""
    v = z.shape[0] // links
    x = torch.view_as_real(z.resolve_conj().reshape(v, links, -1))
    if layout == "soa":
        return x.permute(1, 2, 0, 3)
    b = int(layout[5:])
    whole, rest = divmod(v, b)
    parts = [x[:whole * b].reshape(whole, b, links, -1, 2).permute(0, 2, 3, 1, 4)]
    if rest:
        parts.append(x[whole * b:].permute(1, 2, 0, 3)[None])
    return parts


# ----------------------------------------------------- prepare, run, work
def _tree(names, f):
    a, b = f[0], f[1]
    if names == "commutator":
        return a.adj() * b - b * a.adj()
    if names == "sum":
        return a * b + f[2] * f[3]
    if names == "nested":
        return a * b * f[2] + 0.5 * f[3]
    if names == "factored":
        return a * (b + f[2]) - f[3]
    return (a * b).adj() * f[2]


_L = [("leaf", i) for i in range(4)]
_AUTOGRAD = {"product": ("mul", _L[0], _L[1]),
             "sum": ("add", ("mul", _L[0], _L[1]), ("mul", _L[2], _L[3])),
             "nested": ("add", ("mul", ("mul", _L[0], _L[1]), _L[2]), ("scale", 0.5, _L[3]))}


def prepare(case, seed):
    op, x = case["op"], _inputs(case, seed)
    s = {"op": op, "case": case, "math": MATH[case.get("math", "default")]}
    if op == "batch":
        s["batch"], s["out"], at = su3s.Batch(), [], 0
        for dims in _batch_dims(case):
            lat = su3s.Lattice(dims)
            f = [_field(lat, c[at:at + lat.volume]) for c in x]
            z = f[0].like()
            s["batch"].add(z, f[0] * f[1] + f[2] * f[3])
            s["out"].append(_views(z))
            at += lat.volume
        s["batch"].build()
        return s
    lat = s["lat"] = su3s.Lattice(_dims(case))
    layout = case.get("layout", "soa")
    if op == "product":
        kind = su3s.VECTOR if case["form"] == "av" else su3s.MATRIX
        a = s["a"] = _field(lat, x[0], su3s.MATRIX, case["links"], case["storage"], layout)
        b = s["b"] = _field(lat, x[1], kind, case["links"], case["storage"], layout)
        s["z"] = b.like()
        s["out"] = _views(s["z"])
        s["form"] = case["form"]
    elif op == "tree":
        s["f"] = [_field(lat, c, layout=layout) for c in x]
        s["z"] = s["f"][0].like()
        s["out"] = _views(s["z"])
        s["tree"] = case["tree"]
    elif op == "autograd":
        s["leaves"] = [_field(lat, c).tensor.requires_grad_() for c in x[:-1]]
        s["grad"] = _field(lat, x[-1]).tensor
        s["tree"] = _AUTOGRAD[case["tree"]]
        s["v"] = lat.volume
    elif op in ("dslash", "solver"):
        s["u"] = _field(lat, x[0], su3s.MATRIX, 4, layout=layout)
        s["p"] = _field(lat, x[1], su3s.VECTOR, 4, layout=layout)
        s["z"] = s["p"].like()
        s["out"] = _views(s["z"])
        if op == "solver":
            s["q"] = s["p"].like()
            s["dot"] = torch.empty(1, dtype=torch.float64, device="cuda")
            s["out"] = [s["out"], _views(s["q"]), s["dot"]]
    elif op == "hop":
        kind = su3s.VECTOR if case["kind"] == "vector" else su3s.MATRIX
        s["u"] = _field(lat, x[0], su3s.MATRIX, 4, layout=layout)
        s["p"] = _field(lat, x[1], kind, 1, layout=layout)
        s["z"] = s["p"].like()
        s["out"] = _views(s["z"])
    else:
        s["canon"] = x[0]
        s["u"] = su3s.Field(lat, su3s.MATRIX, 4, PREC[case["storage"]])
        s["z"] = s["u"].like()
        s["out"] = _views(s["z"])
    return s


def run(s):
    op = s["op"]
    if op == "product":
        a, b, form = s["a"], s["b"], s["form"]
        e = a.adj() * b if form == "adj(a)b" else a * b.adj() if form == "a adj(b)" else a * b
        su3s.evaluate(s["z"], e, s["math"])
    elif op == "tree":
        su3s.evaluate(s["z"], _tree(s["tree"], s["f"]), s["math"])
    elif op == "batch":
        s["batch"].launch()
    elif op == "autograd":
        z = su3s.lattice_expr(s["tree"], s["lat"], s["leaves"])
        grads = torch.autograd.grad(z, s["leaves"], s["grad"])
        return [t.detach().view(1, 9, -1, 2)[:, :, :s["v"]] for t in (z,) + grads]
    elif op == "dslash":
        su3s.dslash(s["z"], s["u"], s["p"], s["math"])
    elif op == "solver":
        su3s.dslash(s["z"], s["u"], s["p"])
        su3s.evaluate(s["q"], -KAPPA * s["z"].expr() + s["p"])
        su3s.redot(s["p"], s["q"], s["dot"])
    elif op == "hop":
        su3s.hop(s["z"], s["u"], s["p"], s["math"])
    else:
        s["u"].pack(s["canon"])
        su3s.reunitarize(s["z"], s["u"])
        return [s["out"], s["z"].unpack()]
    return s["out"]


def work(case):
    op, v = case["op"], _volume(case)
    if op == "product":
        r = REAL_BYTES[case["storage"]]
        mat = 12 if "c12" in case["storage"] else 18
        n = v * case["links"]
        if case["form"] == "av":
            return {"bytes": n * r * (18 + 6 + 6), "flops": 66 * n}
        return {"bytes": n * r * 3 * mat, "flops": 198 * n}
    if op == "tree":
        names, flops = TREES[case["tree"]]
        return {"bytes": 144 * v * (len(names) + 1), "flops": flops * v}
    if op == "batch":
        n = sum(d[0] * d[1] * d[2] * d[3] for d in _batch_dims(case))
        return {"bytes": 720 * n, "flops": 414 * n}
    if op == "autograd":
        # forward: leaves read, z written; backward: leaves and dL/dz read, gradients written
        leaves, flops = {"product": (2, 594), "sum": (4, 1206), "nested": (4, 1440)}[case["tree"]]
        return {"bytes": 144 * v * (leaves + 1 + 2 * leaves + 1), "flops": flops * v}
    if op == "dslash":
        return {"bytes": 960 * v, "flops": 1320 * v}
    if op == "solver":
        # D p, then q from both and the product with p while they are at hand
        return {"bytes": (960 + 192) * v, "flops": (1320 + 48 + 48) * v}
    if op == "hop":
        return ({"bytes": 672 * v, "flops": 570 * v} if case["kind"] == "vector"
                else {"bytes": 864 * v, "flops": 1710 * v})
    r = REAL_BYTES[case["storage"]]
    return {"bytes": 4 * v * 2 * (144 + 18 * r), "flops": 4 * v * 700}


# ------------------------------------------------------- 64-bit references
def _cplx(canon):
    return torch.view_as_complex(canon.contiguous())


def _mm(x, y):
    """Batched 3x3 products, column by column."""
    return torch.stack([(x * y[:, None, :, k]).sum(2) for k in range(y.shape[2])], 2)


def _mv(x, y):
    return (x * y[:, None, :]).sum(2)


def _dag(x):
    return x.transpose(1, 2).conj()


def _shift(x, dims, mu, step):
    """x(site + step mu) of an array whose first index is the site (x fastest)."""
    lx, ly, lz, lt = dims
    y = x.reshape(lt, lz, ly, lx, *x.shape[1:])
    return torch.roll(y, -step, 3 - mu).reshape(x.shape)


def _gamma():
    i = 1j
    s = [[[0, i], [i, 0]], [[0, -1], [1, 0]], [[i, 0], [0, -i]], [[1, 0], [0, 1]]]
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    for mu in range(4):
        m = torch.tensor(s[mu], dtype=torch.complex128)
        g[mu, :2, 2:] = m
        g[mu, 2:, :2] = m.conj().T
    return g.cuda()


def _dslash(u, psi, dims):
    """u (V, 4, 3, 3), psi (V, 4, 3): the full 4x4 spin matrices on U psi, nothing projected."""
    one, gam = torch.eye(4, dtype=torch.complex128, device="cuda"), _gamma()
    out = torch.zeros_like(psi)
    for mu in range(4):
        fwd = torch.stack([_mv(u[:, mu], _shift(psi[:, k], dims, mu, 1)) for k in range(4)], 1)
        out += torch.einsum("st,vtc->vsc", one - gam[mu], fwd)
        ub = _dag(_shift(u[:, mu], dims, mu, -1))
        bwd = torch.stack([_mv(ub, _shift(psi[:, k], dims, mu, -1)) for k in range(4)], 1)
        out += torch.einsum("st,vtc->vsc", one + gam[mu], bwd)
    return out


def _rows(z, storage):
    return z[:, :2] if "c12" in storage else z


def _project(m):
    rows = []
    for i in range(3):
        r = m[:, i]
        for _ in range(2):
            for p in rows:
                r = r - (p.conj() * r).sum(1, keepdim=True) * p
        rows.append(r / r.abs().square().sum(1, keepdim=True).sqrt())
    det = (rows[0] * torch.linalg.cross(rows[1], rows[2])).sum(1)
    phase = torch.polar(torch.ones_like(det.real), -det.angle() / 3)
    return torch.stack(rows, 1) * phase[:, None, None]


def exact(case, seed):
    op, x = case["op"], _inputs(case, seed)
    dims, v, layout = _dims(case), _volume(case), case.get("layout", "soa")
    if op == "product":
        m = [_cplx(c) for c in x]
        for k in range(2):
            if "c12" in case["storage"]:
                m[k] = torch.stack((m[k][:, 0], m[k][:, 1], torch.linalg.cross(m[k][:, 0], m[k][:, 1]).conj()), 1)
        a, b = m
        z = (_mv(a, b) if case["form"] == "av" else _mm(_dag(a), b) if case["form"] == "adj(a)b"
             else _mm(a, _dag(b)) if case["form"] == "a adj(b)" else _mm(a, b))
        if case["form"] != "av":
            z = _rows(z, case["storage"])
        return _laid_out(z, case, case["links"], layout)
    if op == "tree":
        f = [_cplx(c) for c in x]
        name = case["tree"]
        if name == "commutator":
            z = _mm(_dag(f[0]), f[1]) - _mm(f[1], _dag(f[0]))
        elif name == "sum":
            z = _mm(f[0], f[1]) + _mm(f[2], f[3])
        elif name == "nested":
            z = _mm(_mm(f[0], f[1]), f[2]) + 0.5 * f[3]
        elif name == "factored":
            z = _mm(f[0], f[1] + f[2]) - f[3]
        else:
            z = _mm(_dag(_mm(f[0], f[1])), f[2])
        return _laid_out(z, case, 1, layout)
    if op == "batch":
        f = [_cplx(c) for c in x]
        z = _mm(f[0], f[1]) + _mm(f[2], f[3])
        sizes = [d[0] * d[1] * d[2] * d[3] for d in _batch_dims(case)]
        return [_laid_out(part, case) for part in torch.split(z, sizes)]
    if op == "autograd":
        f, g = [_cplx(c) for c in x[:-1]], _cplx(x[-1])
        if case["tree"] == "product":
            out = [_mm(f[0], f[1]), _mm(g, _dag(f[1])), _mm(_dag(f[0]), g)]
        elif case["tree"] == "sum":
            out = [_mm(f[0], f[1]) + _mm(f[2], f[3])]
            for k in (0, 2):
                out += [_mm(g, _dag(f[k + 1])), _mm(_dag(f[k]), g)]
        else:
            ab = _mm(f[0], f[1])
            gab = _mm(g, _dag(f[2]))
            out = [_mm(ab, f[2]) + 0.5 * f[3], _mm(gab, _dag(f[1])), _mm(_dag(f[0]), gab),
                   _mm(_dag(ab), g), 0.5 * g]
        return [_laid_out(z, case) for z in out]
    if op in ("dslash", "solver"):
        psi = _cplx(x[1]).reshape(v, 4, 3)
        z = _dslash(_cplx(x[0]).reshape(v, 4, 3, 3), psi, dims)
        first = _laid_out(z.reshape(4 * v, 3), case, 4, layout)
        if op == "dslash":
            return first
        q = psi - KAPPA * z
        dot = (torch.view_as_real(psi) * torch.view_as_real(q)).sum()
        return [first, _laid_out(q.reshape(4 * v, 3), case, 4), dot.reshape(1)]
    if op == "hop":
        u, p = _cplx(x[0]).reshape(v, 4, 3, 3), _cplx(x[1])
        mul = _mv if case["kind"] == "vector" else _mm
        z = torch.zeros_like(p)
        for mu in range(4):
            z += mul(u[:, mu], _shift(p, dims, mu, 1))
            z += mul(_dag(_shift(u[:, mu], dims, mu, -1)), _shift(p, dims, mu, -1))
        return _laid_out(z, case, 1, layout)
    z = _project(_cplx(_stored(x[0], case["storage"])))
    first = _laid_out(z, case, 4)
    return [first, torch.view_as_real(z.contiguous())]
