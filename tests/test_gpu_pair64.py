"""GPU tests of the FP64 pair kernel's group shapes: sizes on both sides of
each change of targets per group (8, 16, 32) and warps per group (1 to 8),
periodic rows of five to nine cells, and lengths in other units
(the kernel finds its pairs in FP32, scaled)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from conftest import assert_atoms

pytestmark = pytest.mark.gpu

# sums of ~1,000 FP64 terms, each rounded to 2^-53: 1e-13 of the RMS, two
# orders to spare
TOL = 1e-11


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def gas(n, box, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.0, 1.0, (n, 3)) * np.asarray(box), rng.uniform(-1.0, 1.0, n)


def evaluate(cfg, pos, q, dev):
    from paper_1402_7216_gb300 import MSM
    plan = MSM(box=cfg["box"], periodic=cfg["periodic"], cutoff=cfg["cutoff"], spacing=cfg["spacing"], order=3,
               splitting=cfg["split"], precision="fp64", max_atoms=len(q))
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    got = [plan.eval(*P), plan.cutoff_eval(*P), plan.wolf_eval(*P, 2.4 / cfg["cutoff"])]
    torch.cuda.synchronize()
    plan.check_status()
    return [(E.item(), phi.cpu().numpy(), F.cpu().numpy()) for E, phi, F in got]


@pytest.mark.parametrize("n,box,periodic,cutoff,split", [
    (9, (20.0, 22.0, 24.0), False, 8.0, 1),
    (1000, (24.0, 22.0, 20.0), True, 8.0, 3),
    (1000, (40.0, 30.0, 35.0), False, 8.0, 2),
    (3649, (33.0, 36.0, 29.0), True, 11.0, 2),
    (9729, (44.0, 47.0, 41.0), True, 8.0, 1),
    (19457, (50.0, 55.0, 61.0), True, 10.0, 2),
    (38913, (60.0, 75.0, 70.0), False, 9.0, 3),
])
def test_group_shapes_match_oracle(n, box, periodic, cutoff, split, dev):
    cfg = dict(box=box, periodic=periodic, cutoff=cutoff, spacing=2.5, split=split)
    pos, q = gas(n, box, seed=n)
    P = O.Params(box=box, periodic=periodic, cutoff=cutoff, spacing=2.5, order=3, split=split)
    ref = [O.msm(P, pos, q), O.cutoff_sum(P, pos, q), O.wolf_sum(P, pos, q, 2.4 / cutoff)]
    for (E, phi, F), r in zip(evaluate(cfg, pos, q, dev), ref):
        assert abs(E - r["E"]) <= TOL * 0.5 * np.abs(q * r["phi"]).sum() + 1e-300
        assert_atoms(F, r["F"], TOL)
        assert_atoms(phi, r["phi"], TOL)


@pytest.mark.parametrize("unit", [2.0 ** -60, 2.0 ** 70])
def test_other_length_units(unit, dev):
    """Lengths scaled by a power of two scale potentials by 1/unit and forces
    by 1/unit^2 (the scaling is exact; the top level's Ewald table is not)."""
    cfg = dict(box=(24.0, 26.0, 23.0), periodic=True, cutoff=8.0, spacing=2.0, split=2)
    pos, q = gas(1500, cfg["box"], seed=5)
    base = evaluate(cfg, pos, q, dev)
    big = dict(cfg, box=tuple(b * unit for b in cfg["box"]), cutoff=8.0 * unit, spacing=2.0 * unit)
    for a, b in zip(base, evaluate(big, pos * unit, q, dev)):
        assert_atoms(b[1] * unit, a[1], TOL)
        assert_atoms(b[2] * unit * unit, a[2], TOL)
