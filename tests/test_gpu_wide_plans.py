"""FP64 products on the wide radix plans (pairs, three and more stages) with
long axes, on both sides of the size up to which FP64 cells take the narrow
plans, and the batched product with the consistent tangent on the members' own
fields (needs a GB300)."""
import numpy as np
import pytest

import oracle
from synth import damage_snapshot, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# Relative RMS error of a product: six transforms of at most 10 levels a line
# and the projection, below 20 eps sqrt(10) = 7e-15 on either side (Higham,
# Accuracy and Stability, 24.1).
TOL = 1.5e-14

# more than 65536 field values: wide plans; each axis long once
WIDE = [(486, 24, 8), (24, 486, 8), (8, 24, 486), (720, 8, 12), (8, 250, 40), (8, 12, 720), (900, 6, 6), (6, 972, 4),
        (4, 6, 1000), (16, 20, 162), (162, 144), (144, 162), (48, 900), (900, 48), (1000, 30), (30, 1000)]
# the last grids on the narrow plans (64800 values) and the first on the wide
# ones (67500, 69120)
EDGE = [(18, 20, 30), (144, 150), (150, 150), (12, 16, 60)]


def _cell(dims, seed):
    rng = np.random.default_rng(seed)
    return (rng.random(tuple(reversed(dims))) < 0.3).astype(np.uint8)


@pytest.mark.parametrize("dims", WIDE + EDGE, ids=lambda d: "x".join(map(str, d)))
def test_fp64_product_matches_oracle(dims):
    from paper_2207_10657_gb300 import Phase, RVESolver, build
    build.build()
    pm = _cell(dims, sum(dims))
    D = damage_snapshot(pm, dmax=0.9, seed=1).astype(np.float64)
    v = random_field(6 if len(dims) == 3 else 3, dims, seed=2)
    s = RVESolver(dims, pm, [Phase(1.0, 0.3, True, 1e-4, 1e-3), Phase(10.0, 0.2)], precision=64)
    s.set_damage(torch.from_numpy(D).cuda())
    got = s.hessp(torch.from_numpy(v).cuda()).cpu().numpy()
    s.close()
    rve = oracle.RVE(pm, [oracle.Phase(1.0, 0.3, True, 1e-4, 1e-3), oracle.Phase(10.0, 0.2)])
    ref = rve.hessp(D, v)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)


def test_batched_consistent_product_matches_single_contexts():
    """One Newton iteration from the unloaded state to well past the damage
    threshold leaves every member unconverged and loading; the batched product
    of that state against single contexts set to it."""
    from paper_2207_10657_gb300 import Phase, RVEBatch, RVESolver, build
    build.build()
    phases = [Phase(1.0, 0.3, True, 1e-4, 1e-3), Phase(10.0, 0.2)]
    dims = [(24, 20), (16, 12, 10), (64, 64), (30, 18, 8)]
    pms = [_cell(d, i) for i, d in enumerate(dims)]
    opts = dict(hessian=1, max_nr=1, R0=1.0, Rmax=1.0)
    b = RVEBatch(dims, pms, phases, **opts)
    nc = [3 if len(d) == 2 else 6 for d in dims]
    b.solve_step([[4e-4] + [0.0] * (n - 1) for n in nc], [[0] * n for n in nc], raise_on_error=False)
    vs = [torch.from_numpy(random_field(n, d, seed=i)).float().cuda() for i, (n, d) in enumerate(zip(nc, dims))]
    outs = b.hessp(vs)
    for i, d in enumerate(dims):
        st = b.get_state(i)
        got = []
        for hessian in (1, 0):
            s = RVESolver(d, pms[i], phases, hessian=hessian)
            s.set_state(st["eps"], st["kappa"])
            got.append(s.hessp(vs[i]).double())
            s.close()
        assert float(st["damage"].max()) > 0.1
        assert float((got[0] - got[1]).norm()) > 1e-2 * float(got[0].norm())  # the tangents differ here
        # FP32 products on two tilings: 20 * 2^-24 * sqrt(10) each (4e-6)
        assert float((outs[i].double() - got[0]).norm()) <= 8e-6 * float(got[0].norm()), d
    b.close()
