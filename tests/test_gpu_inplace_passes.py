"""The generic (runtime-length) passes at the lengths where their in-place
transforms can go wrong: single-stage lengths, every radix and radix pair,
three and more stages, remainder columns shared between planes, lines that
fill a block alone; Hessian-vector products against the FP64 oracle (needs a
GB300)."""
import numpy as np
import pytest

import oracle
from synth import damage_snapshot, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# An FFT's relative RMS error grows as eps sqrt(log2 N) times a small constant
# (Higham, Accuracy and Stability, 24.1); six transforms of at most 10 levels
# and the projection stay below 20 eps: FP32 20 * 2^-24 * sqrt(10) ~ 4e-6.
TOL = {32: 5e-6, 64: 1e-14}

GRIDS = [
    (2, 6, 4), (10, 2, 12), (16, 18, 20), (30, 36, 24), (40, 50, 6), (54, 12, 60), (90, 72, 10), (4, 100, 48),
    (6, 4, 162), (2, 250, 8), (150, 4, 2), (2, 2, 486), (486, 2, 4), (1000, 2, 2), (2, 972, 2), (2, 2, 1000),
    (12, 10), (50, 90), (162, 24), (2, 720), (900, 6), (18, 1000),
]


def _cell(dims, seed):
    rng = np.random.default_rng(seed)
    return (rng.random(tuple(reversed(dims))) < 0.3).astype(np.uint8)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("dims", GRIDS, ids=lambda d: "x".join(map(str, d)))
def test_product_matches_oracle(dims, precision):
    from paper_2207_10657_gb300 import Phase, RVESolver, build
    build.build()
    pm = _cell(dims, sum(dims))
    D = damage_snapshot(pm, dmax=0.9, seed=1).astype(np.float64)
    v = random_field(6 if len(dims) == 3 else 3, dims, seed=2)
    dt = torch.float32 if precision == 32 else torch.float64
    s = RVESolver(dims, pm, [Phase(1.0, 0.3, True, 1e-4, 1e-3), Phase(10.0, 0.2)], precision=precision, passes=1)
    Dt, vt = torch.from_numpy(D).to(dt).cuda(), torch.from_numpy(v).to(dt).cuda()
    s.set_damage(Dt)
    got = s.hessp(vt).double().cpu().numpy()
    s.close()
    rve = oracle.RVE(pm, [oracle.Phase(1.0, 0.3, True, 1e-4, 1e-3), oracle.Phase(10.0, 0.2)])
    ref = rve.hessp(Dt.double().cpu().numpy(), vt.double().cpu().numpy())
    assert np.linalg.norm(got - ref) <= TOL[precision] * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [1, 33, 256])
def test_batched_product_in_place_of_many_members(n):
    """Work lists of one, of a little more than a warp's and of the largest
    number of members; the products overwrite their inputs."""
    from paper_2207_10657_gb300 import Phase, RVEBatch, RVESolver, build
    from paper_2207_10657_gb300 import binding as B
    build.build()
    phases = [Phase(1.0, 0.3, True, 1e-4, 1e-3), Phase(10.0, 0.2)]
    kinds = [(8, 6), (10, 4, 6), (12, 18)]
    dims = [kinds[i % 3] for i in range(n)]
    pms = [_cell(d, i) for i, d in enumerate(dims)]
    Ds = [torch.from_numpy(damage_snapshot(pm, dmax=0.9, seed=i)).float().cuda() for i, pm in enumerate(pms)]
    vs = [torch.from_numpy(random_field(6 if len(d) == 3 else 3, d, seed=i)).float().cuda()
          for i, d in enumerate(dims)]
    ref = []
    for d, pm, D, v in zip(dims, pms, Ds, vs):
        s = RVESolver(d, pm, phases, passes=1)
        s.set_damage(D)
        ref.append(s.hessp(v))
        s.close()
    b = RVEBatch(dims, pms, phases)
    for i, D in enumerate(Ds):
        b.set_damage(i, D)
    B.rve_batch_hessp(b.h, [v.data_ptr() for v in vs], [v.data_ptr() for v in vs])
    torch.cuda.synchronize()
    for got, want in zip(vs, ref):
        assert float((got - want).norm()) <= TOL[32] * float(want.norm())
    with pytest.raises(B.RveError):
        B.rve_batch_hessp(b.h, [0] * n, [v.data_ptr() for v in vs])
    b.close()
