"""Timed cases of the framework: what its users run, over the sizes, element types and options it serves.

Kinds of case (``case["kind"]``)

* ``hv``    one Hessian-vector product G : (tangent : v) on a context with a damage snapshot, the step that every
            load path, L-BFGS iteration and effective-stiffness solve repeats (``RVESolver.hessp``).  Options: field
            type FP32 / FP64, the symmetric consistent tangent at a loading state, Kuhn simplices.
* ``batch`` one batched product of many cells of uneven sizes (``RVEBatch.hessp``).
* ``step``  one whole load increment from the unloaded cell (``RVESolver.solve_step``): Newton, Steihaug CG,
            constitutive update, ratio test; the strain, stress and damage fields are returned.
* ``fno``   forward and backward pass of the learned warm start's network on one training batch
            (``SpectralOperator.loss_grad``), with the gradient of every parameter returned.

Fields are component-major, Mandel components, x fastest; a grid is given as its sizes (nx, ny[, nz]).
"""
import math

import numpy as np
import torch

from paper_2207_10657_gb300 import Phase, RVEBatch, RVESolver
from paper_2207_10657_gb300.learned import SpectralOperator

# E, nu, damaging, kappa0, kappaf of the damaging matrix and the stiff inclusions
MATRIX = (1.0, 0.3, True, 1e-4, 1e-3)
STIFF = (10.0, 0.2, False, 0.0, 0.0)
FREE_ZZ = (1, 1, 0, 1, 1, 1)  # uniaxial eps_zz: every other mean component is stress-free
SQ2 = math.sqrt(2.0)


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest cell: 32^2 plane strain with a disc, all-FP64; bound by launches and by how few blocks run
        _hv("hv2d_32_f64", 32, 32, dtype="f64"),
        # the largest 2D cell of the batched study, alone
        _hv("hv2d_512_f32", 512, 512),
        # the 128^3 sphere cell of the uniaxial load path
        _hv("hv3d_128_f32", 128, 128, 128),
        # the 256^3 sphere cell: the benchmark's product
        _hv("hv3d_256_f32", 256, 256, 256),
        # the largest cell of the size study
        _hv("hv3d_384_f32", 384, 384, 384),
        # a cell whose sides follow a specimen and not a power of two: three different 5-smooth lengths
        _hv("hv3d_160x120x90_f32", 160, 120, 90),
        # the all-FP64 arm of the precision study
        _hv("hv3d_128_f64", 128, 128, 128, dtype="f64"),
        # the consistent tangent at a state past the damage onset, at an evaluation size of the warm start
        _hv("hv3d_192_consistent_f32", 192, 192, 192, consistent=True),
        # Kuhn tetrahedra, six strain points per voxel
        _hv("hv3d_64_tetrahedra_f32", 64, 64, 64, simplex=True),
        # 96 cells of uneven sizes, half 2D from 64^2 to 512^2, half 3D from 32^3 to 96^3
        {"name": "batch_96_f32", "kind": "batch", "members": 96, "draw": 0},
        # one elastic increment (1e-5, as the warm start's load paths take) of the 256^3 cell, from call to converged state
        {"name": "step_256_f32", "kind": "step", "nx": 256, "ny": 256, "nz": 256, "strain": 1e-5},
        # one training batch of the warm start's network: four 64^3 samples
        {"name": "fno_train_64", "kind": "fno", "n": 64, "batch": 4, "layers": 4, "modes": 8},
    ]


def _hv(name, nx, ny, nz=0, dtype="f32", consistent=False, simplex=False):
    return {"name": name, "kind": "hv", "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "consistent": consistent,
            "simplex": simplex}


def _sizes(lo, hi):
    """Even numbers in [lo, hi] with no prime factor above 5: the lengths an axis may have."""
    out = []
    for n in range(lo + (lo & 1), hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _pick(rng, lo, hi):
    """An allowed length, spread over the logarithm of [lo, hi]."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_sizes(lo, hi), key=lambda n: abs(math.log(n / t)))


def draw(rng):
    kind = rng.choice(("hv2d", "hv3d", "hv3d", "hv3d", "hv3d64", "consistent", "simplex", "batch", "step", "fno"))
    if kind == "hv2d":
        return _unnamed(_hv("", _pick(rng, 32, 512), _pick(rng, 32, 512), dtype=rng.choice(("f32", "f64"))))
    if kind == "hv3d":
        if rng.random() < 0.4:  # a cube of a power of two or three times one, as most cells are
            n = rng.choice((32, 64, 96, 128, 192, 256, 384))
            return _unnamed(_hv("", n, n, n if n in (32, 64, 96, 192) else rng.choice((32, 48, 64, 96))))
        return _unnamed(_hv("", _pick(rng, 32, 300), _pick(rng, 32, 300), _pick(rng, 32, 300)))
    if kind == "hv3d64":
        return _unnamed(_hv("", _pick(rng, 32, 128), _pick(rng, 32, 128), _pick(rng, 32, 128), dtype="f64"))
    if kind == "consistent":
        n = rng.choice((64, 96, 128, 192))
        return _unnamed(_hv("", n, rng.choice((64, 90, 128)), rng.choice((32, 72, 128)), consistent=True))
    if kind == "simplex":
        if rng.random() < 0.5:
            return _unnamed(_hv("", _pick(rng, 32, 512), _pick(rng, 32, 512), simplex=True))
        return _unnamed(_hv("", _pick(rng, 24, 80), _pick(rng, 24, 80), _pick(rng, 24, 80), simplex=True))
    if kind == "batch":
        return {"kind": "batch", "members": rng.choice((8, 17, 32, 48, 96)), "draw": rng.randrange(1, 1 << 20)}
    if kind == "step":
        n = [_pick(rng, 32, 160) for _ in range(3)]
        return {"kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "strain": rng.choice((5e-6, 1e-5))}
    return {"kind": "fno", "n": rng.choice((32, 48, 64)), "batch": rng.choice((1, 2, 4)),
            "layers": rng.choice((2, 4)), "modes": rng.choice((4, 6, 8))}


def _unnamed(case):
    del case["name"]
    return case


# ----------------------------------------------------------------- inputs
def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + k)


def _dims(case):
    return tuple(case[a] for a in ("nx", "ny", "nz") if case[a])


def _inclusions(dims, frac, rmin, rmax, rng):
    """Phase map with randomly placed discs / spheres (phase 1), periodic, up to about the volume fraction `frac`."""
    nd = len(dims)
    shape = tuple(reversed(dims))
    ph = np.zeros(shape, np.uint8)
    filled, goal = 0.0, frac * float(np.prod(dims))
    while filled < goal:
        r = rng.uniform(rmin, rmax)
        c = rng.uniform(0, 1, nd) * np.asarray(dims)
        ax = [np.arange(math.floor(c[a] - r), math.ceil(c[a] + r) + 1) for a in range(nd)]
        d2 = 0.0
        for a in range(nd):
            v = [1] * nd
            v[nd - 1 - a] = -1
            d2 = d2 + ((ax[a] + 0.5 - c[a]) ** 2).reshape(v)
        inside = d2 <= r * r
        if all(i <= n for i, n in zip(inside.shape, shape)):
            idx = np.ix_(*[ax[a] % dims[a] for a in reversed(range(nd))])
            ph[idx] |= inside.astype(np.uint8)
        filled += (4.0 / 3.0 * math.pi * r ** 3) if nd == 3 else math.pi * r * r
    return ph


def _cell(dims, seed, frac=None):
    """A cell's phase map: discs (2D) at 30 % or spheres (3D) of the load paths' relative sizes at 5 %."""
    rng = np.random.default_rng(seed)
    n = min(dims)
    if len(dims) == 2:
        return _inclusions(dims, 0.3 if frac is None else frac, n / 32, n / 10, rng)
    return _inclusions(dims, 0.05 if frac is None else frac, max(2.0, n / 32), max(3.0, n / 12), rng)


def _phases():
    return [Phase(*MATRIX), Phase(*STIFF)]


def _hv_data(case, seed):
    """Phase map, damage snapshot (or loading state) and the vector of one `hv` case, as FP64-exact tensors of the
    case's type."""
    dims = _dims(case)
    shape = tuple(reversed(dims))
    nc = 6 if len(dims) == 3 else 3
    nq = (6 if nc == 6 else 2) if case["simplex"] else 1
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    ph = torch.from_numpy(_cell(dims, seed)).cuda()
    g = _gen(seed)
    pts = (nq,) if nq > 1 else ()
    d = {"dims": dims, "ph": ph, "v": torch.randn((nc,) + pts + shape, generator=g, device="cuda", dtype=dt)}
    if case["consistent"]:
        # a state well inside the softening range: kappa between 1.2 and 4 kappa0 everywhere, loading on about half
        # of the matrix (history below the state's kappa), unloading on the rest
        eps = torch.randn((nc,) + shape, generator=g, device="cuda", dtype=torch.float64)
        want = 1e-4 * (1.2 + 2.8 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64))
        eps[0] += 6  # tension along x everywhere
        eps = (eps * (want / _positive(eps)[1])).to(dt)
        lo = torch.rand(shape, generator=g, device="cuda") < 0.5
        kh = torch.where(lo, 5e-5, 5e-4).to(dt) * (ph == 0)
        d.update(eps=eps, kh=kh)
    else:
        D = 0.9 * torch.rand(pts + shape, generator=g, device="cuda", dtype=dt)
        d["D"] = D * (ph == 0).to(dt)
    return d


def _batch_data(case, seed):
    rng = np.random.default_rng(7 + case["draw"])
    m = case["members"]
    s2, s3 = _sizes(64, 512), _sizes(32, 96)
    members = []
    for k in range(m):
        n = int(rng.choice(s2 if k < m // 2 else s3))
        dims = (n, n) if k < m // 2 else (n, n, n)
        frac = float(rng.uniform(0.1, 0.4) if k < m // 2 else rng.uniform(0.1, 0.3))
        members.append((dims, frac))
    g = _gen(seed)
    out = []
    for k, (dims, frac) in enumerate(members):
        shape = tuple(reversed(dims))
        ph = torch.from_numpy(_cell(dims, (seed, k), frac)).cuda()
        D = 0.9 * torch.rand(shape, generator=g, device="cuda") * (ph == 0)
        v = torch.randn((3 if len(dims) == 2 else 6,) + shape, generator=g, device="cuda")
        out.append((dims, ph, D, v))
    return out


def _fno_data(case, seed):
    n, b = case["n"], case["batch"]
    g = _gen(seed)
    X = torch.randn((b, n, n, n, 16), generator=g, device="cuda")
    X[..., :2] = torch.nn.functional.one_hot((X[..., 0] > 1.0).long(), 2).float()
    T = torch.randn((b, n, n, n, 6), generator=g, device="cuda")
    rng = np.random.default_rng(seed)
    w, m = 32, case["modes"]
    par = [rng.standard_normal((16, w)) / 4, 0.1 * rng.standard_normal(w)]
    for _ in range(case["layers"]):
        par += [rng.standard_normal((w, w)) / math.sqrt(w), 0.1 * rng.standard_normal(w),
                rng.standard_normal((m ** 3, 2 * w, 2 * w), dtype=np.float32) / (2 * w)]
    par += [rng.standard_normal((w, 6)) / math.sqrt(w), 0.1 * rng.standard_normal(6)]
    return X, T, [np.asarray(p, dtype=np.float32) for p in par]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "hv":
        d = _hv_data(case, seed)
        s = RVESolver(d["dims"], d["ph"], _phases(), precision=64 if case["dtype"] == "f64" else 32,
                      hessian=int(case["consistent"]), element=int(case["simplex"]))
        if case["consistent"]:
            s.set_state(d["eps"], d["kh"])
        else:
            s.set_damage(d["D"])
        return {"kind": kind, "solver": s, "v": d["v"], "out": s.field()}
    if kind == "batch":
        data = _batch_data(case, seed)
        b = RVEBatch([m[0] for m in data], [m[1] for m in data], _phases())
        for i, m in enumerate(data):
            b.set_damage(i, m[2])
        return {"kind": kind, "batch": b, "v": [m[3] for m in data]}
    if kind == "step":
        dims = _dims(case)
        s = RVESolver(dims, torch.from_numpy(_cell(dims, seed)).cuda(), _phases())
        return {"kind": kind, "solver": s, "zero": s.field(0.0), "dE": [0, 0, case["strain"], 0, 0, 0]}
    X, T, par = _fno_data(case, seed)
    net = SpectralOperator(layers=case["layers"], modes=case["modes"])
    net.set_params(np.concatenate([p.ravel() for p in par]))
    return {"kind": kind, "net": net, "X": X, "T": T, "dims": (case["n"],) * 3}


def run(state):
    kind = state["kind"]
    if kind == "hv":
        return state["solver"].hessp(state["v"], out=state["out"])
    if kind == "batch":
        # 2D and 3D members, each as one flat vector (many members, few outputs)
        outs = state["batch"].hessp(state["v"])
        return {f"cells_{d}d": torch.cat([o.reshape(-1) for o in outs if o.dim() == d + 1]) for d in (2, 3)}
    if kind == "step":
        s = state["solver"]
        s.set_state(state["zero"])
        rep = s.solve_step(state["dE"], free_mask=FREE_ZZ)
        st = s.get_state()
        return {"eps": st["eps"], "sigma": st["sigma"], "damage": st["damage"],
                "mean_stress_zz": float(rep["mean_stress"][2]), "mean_strain": np.array(rep["mean_strain"])}
    loss = state["net"].loss_grad(state["X"], state["T"], state["dims"])
    return {"loss": loss, "grad": state["net"].get_params(want_grad=True)[1]}


# ------------------------------------------------------------------- work
def _transform_flops(dims, lines):
    """Real forward and inverse FFT of `lines` lines per voxel."""
    n = float(np.prod(dims))
    return 2 * 2.5 * n * math.log2(n) * lines


def _hv_work(dims, es, nq=1, consistent=False):
    n, nc = float(np.prod(dims)), 6 if len(dims) == 3 else 3
    by = n * nq * es * (2 * nc + 1) + n  # vector in, product out, damage, phase
    if consistent:
        by += n * es * (1 + nc)  # the loading half's C:eps and n, D'
    return {"bytes": by, "flops": _transform_flops(dims, nc * nq) + 60.0 * n * nq}


def work(case):
    if case["kind"] == "hv":
        dims = _dims(case)
        nq = (6 if len(dims) == 3 else 2) if case["simplex"] else 1
        return _hv_work(dims, 8 if case["dtype"] == "f64" else 4, nq, case["consistent"])
    if case["kind"] == "batch":
        rng = np.random.default_rng(7 + case["draw"])
        m = case["members"]
        s2, s3 = _sizes(64, 512), _sizes(32, 96)
        tot = {"bytes": 0.0, "flops": 0.0}
        for k in range(m):
            n = int(rng.choice(s2 if k < m // 2 else s3))
            rng.uniform()
            w = _hv_work((n, n) if k < m // 2 else (n, n, n), 4)
            tot = {q: tot[q] + w[q] for q in tot}
        return tot
    if case["kind"] == "step":
        dims = _dims(case)
        n = float(np.prod(dims))
        # start state, phases in; strain, stress, damage, history out; at least one gradient and one product
        return {"bytes": n * (4 * (3 * 6 + 3) + 1), "flops": 2 * (_transform_flops(dims, 6) + 60.0 * n)}
    n, b, m = case["n"], case["batch"], case["modes"]
    vox, w = float(b * n ** 3), 32
    par = case["layers"] * m ** 3 * 4 * w * w
    # 1x1 mixes forward and twice backward; truncated transforms as products along the axes (x dominates)
    mix = 2 * vox * w * (16 + 6 + case["layers"] * w)
    dft = case["layers"] * 2 * (2 * vox * 2 * m * w)
    return {"bytes": vox * 4 * (16 + 6) + 4.0 * 2 * par, "flops": 3 * mix + 2 * dft + 6.0 * b * par}


# ------------------------------------------- the same results in 64 bits
def _ref_solver_tables(dims):
    """e^{i theta} - 1 and (1 + e^{i theta}) / 2 per axis x, y[, z], shaped for a half spectrum over x."""
    nd = len(dims)
    diff, avg = [], []
    for a, n in enumerate(dims):
        k = torch.arange(n // 2 + 1 if a == 0 else n, device="cuda", dtype=torch.float64)
        e = torch.polar(torch.ones_like(k), 2 * math.pi * k / n)
        d, m = e - 1, (1 + e) / 2
        d[0] = 0
        if n // 2 < len(m):
            m[n // 2] = 0
        v = [1] * nd
        v[nd - 1 - a] = -1
        diff.append(d.reshape(v))
        avg.append(m.reshape(v))
    return diff, avg


def _ref_project(x, dims, free=None):
    """G : x in FP64 for the one-element-per-voxel gradient; x (ncomp, *grid)."""
    nd = len(dims)
    axes = tuple(range(1, nd + 1))
    z = torch.fft.rfftn(x.double(), dim=axes)
    mean = z[(slice(None),) + (0,) * nd].clone()
    diff, avg = _ref_solver_tables(dims)
    D = []
    for a in range(nd):
        t = diff[a]
        for b in range(nd):
            if b != a:
                t = t * avg[b]
        D.append(t.expand(z.shape[1:]) if t.shape != z.shape[1:] else t)
    n2 = sum(t.real ** 2 + t.imag ** 2 for t in D)
    inv = torch.where(n2 > 0, 1 / torch.where(n2 > 0, n2, 1.0), 0.0)
    pos = {(0, 0): 0, (1, 1): 1, (0, 1): 2} if nd == 2 else \
        {(0, 0): 0, (1, 1): 1, (2, 2): 2, (1, 2): 3, (0, 2): 4, (0, 1): 5}

    def comp(i, j):
        c = pos[(min(i, j), max(i, j))]
        return z[c] if i == j else z[c] / SQ2
    w = []
    for i in range(nd):
        w.append(sum(comp(i, j) * D[j].conj() for j in range(nd)))
    s = sum(w[i] * D[i].conj() for i in range(nd)) * (-0.5 * inv)
    w = [w[i] + s * D[i] for i in range(nd)]
    for (i, j), c in pos.items():
        z[c] = 2 * inv * D[i] * w[i] if i == j else SQ2 * inv * (D[i] * w[j] + D[j] * w[i])
    for c in range(len(z)):
        z[(c,) + (0,) * nd] = mean[c] if free is not None and free[c] else 0
    return torch.fft.irfftn(z, s=x.shape[1:], dim=axes)


def _lame(ph):
    out = []
    for k in (0, 1):
        E, nu = (MATRIX, STIFF)[k][:2]
        out.append((E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))))
    m = (ph == 1).double()
    return tuple(out[0][q] + (out[1][q] - out[0][q]) * m for q in (0, 1))


def _elastic(v, ph):
    """C : v per point; v (ncomp, [nq,] *grid)."""
    lam, mu = _lame(ph)
    nd = 2 if len(v) == 3 else 3
    out = 2 * mu * v
    tr = lam * v[:nd].sum(0)
    out[:nd] += tr
    return out


def _positive(e):
    """Positive part (Mandel) of a symmetric 3 x 3 field and its norm, by Jacobi rotations in FP64."""
    e = e.double()
    A = [[None] * 3 for _ in range(3)]
    for i in range(3):
        A[i][i] = e[i].clone()
    for c, (i, j) in ((3, (1, 2)), (4, (0, 2)), (5, (0, 1))):
        A[i][j] = e[c] / SQ2
        A[j][i] = A[i][j]
    one, zero = torch.ones_like(e[0]), torch.zeros_like(e[0])
    V = [[one if i == j else zero for j in range(3)] for i in range(3)]
    for _ in range(7):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            small = A[p][q].abs() < 1e-300
            th = (A[q][q] - A[p][p]) / (2 * torch.where(small, 1.0, A[p][q]))
            t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + torch.sqrt(th * th + 1))
            t = torch.where(small, 0.0, t)
            c = 1 / torch.sqrt(t * t + 1)
            s = t * c
            for k in range(3):
                A[k][p], A[k][q] = c * A[k][p] - s * A[k][q], s * A[k][p] + c * A[k][q]
            for k in range(3):
                A[p][k], A[q][k] = c * A[p][k] - s * A[q][k], s * A[p][k] + c * A[q][k]
            for k in range(3):
                V[k][p], V[k][q] = c * V[k][p] - s * V[k][q], s * V[k][p] + c * V[k][q]
    lam = [A[k][k].clamp_min(0) for k in range(3)]
    out = []
    for i, j, f in ((0, 0, 1), (1, 1, 1), (2, 2, 1), (1, 2, SQ2), (0, 2, SQ2), (0, 1, SQ2)):
        out.append(f * sum(lam[k] * V[i][k] * V[j][k] for k in range(3)))
    return torch.stack(out), torch.sqrt(sum(x * x for x in lam))


def _ref_simplex(x, dims):
    """G : x in FP64 for Kuhn simplices, every mean component controlled; x (ncomp, nq, *grid)."""
    import itertools
    nd = len(dims)
    axes = tuple(range(2, nd + 2))
    z = torch.fft.rfftn(x, dim=axes)
    diff, _ = _ref_solver_tables(dims)
    perms = list(itertools.permutations(range(nd)))
    pairs = [(0, 0), (1, 1), (0, 1)] if nd == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
    sym = []
    for pi in perms:
        pre, D = torch.ones((), dtype=torch.complex128, device="cuda"), [None] * nd
        for a in pi:
            D[a] = (pre * diff[a]).expand(z.shape[2:])
            pre = pre * (diff[a] + 1)
        sym.append(D)
    M = [[0.0] * nd for _ in range(nd)]
    b = [0.0] * nd

    def rows(D):
        for c, (i, j) in enumerate(pairs):
            yield c, ({i: D[i]} if i == j else {j: D[i] / SQ2, i: D[j] / SQ2})
    for q, D in enumerate(sym):
        for c, r in rows(D):
            for i, ri in r.items():
                b[i] = b[i] + ri.conj() * z[c, q]
                for j, rj in r.items():
                    M[i][j] = M[i][j] + ri.conj() * rj
    Mt = torch.stack([torch.stack(r, -1) for r in M], -2)
    bt = torch.stack(b, -1)
    at0 = (0,) * nd
    Mt[at0] = torch.eye(nd, dtype=Mt.dtype, device="cuda")
    bt[at0] = 0
    if nd == 2:
        det = Mt[..., 0, 0] * Mt[..., 1, 1] - Mt[..., 0, 1] * Mt[..., 1, 0]
        a = [(bt[..., 0] * Mt[..., 1, 1] - bt[..., 1] * Mt[..., 0, 1]) / det,
             (bt[..., 1] * Mt[..., 0, 0] - bt[..., 0] * Mt[..., 1, 0]) / det]
    else:
        col = [Mt[..., :, k] for k in range(3)]
        cr = torch.linalg.cross
        det = (col[0] * cr(col[1], col[2])).sum(-1)
        a = [(bt * cr(col[(k + 1) % 3], col[(k + 2) % 3])).sum(-1) / det for k in range(3)]
    for q, D in enumerate(sym):
        for c, r in rows(D):
            z[c, q] = sum(ri * a[i] for i, ri in r.items())
    z[(slice(None), slice(None)) + at0] = 0
    return torch.fft.irfftn(z, s=x.shape[2:], dim=axes)


def _ref_hv(v, ph, D, dims):
    return _ref_project((1 - D.double()) * _elastic(v.double(), ph), dims)


def _exact_hv(case, seed):
    d = _hv_data(case, seed)
    v = d["v"].double()
    if case["simplex"]:
        return _ref_simplex((1 - d["D"].double()) * _elastic(v, d["ph"]), d["dims"])
    if not case["consistent"]:
        return _ref_hv(v, d["ph"], d["D"], d["dims"])
    eps, kh = d["eps"].double(), d["kh"].double()
    ep, kt = _positive(eps)
    mat = d["ph"] == 0
    k0, kf = np.float64(np.float32(MATRIX[3])), np.float64(np.float32(MATRIX[4]))
    k = torch.maximum(kt, kh)
    D = torch.where(mat & (k > k0), kf * (k - k0) / (k * (kf - k0)), 0.0)
    dp = torch.where(mat & (kt > kh) & (k > k0) & (k < kf), kf * k0 / (k * k * (kf - k0)), 0.0)
    Ce, n = _elastic(eps, d["ph"]), ep / kt
    s = (1 - D) * _elastic(v, d["ph"]) - 0.5 * dp * (Ce * (n * v).sum(0) + n * (Ce * v).sum(0))
    return _ref_project(s, d["dims"])


def _exact_step(case, seed):
    """The elastic increment's exact solution: conjugate gradients on G:C:(E + x) = 0 to 1e-12."""
    dims = _dims(case)
    ph = torch.from_numpy(_cell(dims, seed)).cuda()
    e = torch.zeros((6,) + tuple(reversed(dims)), dtype=torch.float64, device="cuda")
    e[2] = case["strain"]
    r = -_ref_project(_elastic(e, ph), dims, FREE_ZZ)
    d, rr = r.clone(), float((r * r).sum())
    stop = 1e-24 * rr
    for _ in range(400):
        if rr <= stop:
            break
        Hd = _ref_project(_elastic(d, ph), dims, FREE_ZZ)
        a = rr / float((d * Hd).sum())
        e += a * d
        r -= a * Hd
        new = float((r * r).sum())
        d = r + (new / rr) * d
        rr = new
    if bool((_positive(e)[1][ph == 0] > MATRIX[3]).any()):
        return None  # not elastic after all
    s = _elastic(e, ph)
    nv = float(np.prod(dims))
    return {"eps": e, "sigma": s, "damage": torch.zeros_like(e[0]), "mean_stress_zz": float(s[2].sum() / nv),
            "mean_strain": (e.reshape(6, -1).sum(1) / nv).cpu().numpy()}


def _exact_fno(case, seed):
    X, T, par = _fno_data(case, seed)
    n, m, w = case["n"], case["modes"], 32
    X, T = X.double(), T.double()
    p = [torch.from_numpy(q).cuda().double().requires_grad_() for q in par]
    iy = (torch.arange(m, device="cuda") - m // 2) % n
    h = X @ p[0] + p[1]
    for l in range(case["layers"]):
        W, b, R = p[2 + 3 * l: 5 + 3 * l]
        H = torch.fft.rfft(h, dim=3)[:, :, :, :m]
        H = torch.fft.fft(H, dim=2)[:, :, iy]
        H = torch.fft.fft(H, dim=1)[:, iy]
        S = torch.cat([H.real, H.imag], -1)
        S = torch.einsum("zyxoi,bzyxi->bzyxo", R.reshape(m, m, m, 2 * w, 2 * w), S)
        Z = torch.complex(S[..., :w].contiguous(), S[..., w:].contiguous())
        # back into the half spectrum, z index by z index
        full = torch.zeros((Z.shape[0], m, n, n // 2 + 1, w), dtype=Z.dtype, device="cuda")
        full = full.index_copy(2, iy, torch.nn.functional.pad(Z, (0, 0, 0, n // 2 + 1 - m)))
        full = torch.zeros((Z.shape[0], n, n, n // 2 + 1, w), dtype=Z.dtype, device="cuda").index_copy(1, iy, full)
        K = torch.fft.irfftn(full, s=(n, n, n), dim=(1, 2, 3))
        u = K + h @ W + b
        h = torch.nn.functional.gelu(u, approximate="tanh") if l < case["layers"] - 1 else u
    loss = ((h @ p[-2] + p[-1] - T) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": torch.cat([q.grad.reshape(-1) for q in p])}


def exact(case, seed):
    if case["kind"] == "hv":
        return _exact_hv(case, seed)
    if case["kind"] == "batch":
        outs = [_ref_hv(v, ph, D, dims) for dims, ph, D, v in _batch_data(case, seed)]
        return {f"cells_{d}d": torch.cat([o.reshape(-1) for o in outs if o.dim() == d + 1]) for d in (2, 3)}
    if case["kind"] == "step":
        return _exact_step(case, seed)
    return _exact_fno(case, seed)
