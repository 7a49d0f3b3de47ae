"""GPU tests of the FP64 pair kernel's dispatch and of its reciprocal square root.

Group shapes: 8 targets and 8, 4, 2 or 1 warps a group up to 1,816, 3,640, 7,288
and 19,440 atoms, then 16 targets: both sides of each line, MSM, cutoff and Wolf
sums against the oracle."""
import decimal
import math

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


@pytest.mark.parametrize("n", [1816, 1817, 3640, 3641, 7288, 7289, 19440, 19441])
def test_group_shapes_match_oracle(n, dev):
    from paper_1402_7216_gb300 import MSM
    periodic = n % 2 == 0
    box = tuple(f * (n / 0.08) ** (1 / 3) for f in (1.0, 1.1, 0.95))
    rng = np.random.default_rng(n)
    pos, q = rng.uniform(0.0, 1.0, (n, 3)) * np.asarray(box), rng.uniform(-1.0, 1.0, n)
    par = dict(box=box, periodic=periodic, cutoff=8.0, spacing=2.5, order=3)
    plan = MSM(splitting=2, precision="fp64", max_atoms=n, **par)
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    got = [plan.eval(*P), plan.cutoff_eval(*P), plan.wolf_eval(*P, 0.3)]
    plan.check_status()
    R = O.Params(split=2, **par)
    for (E, phi, F), r in zip(got, [O.msm(R, pos, q), O.cutoff_sum(R, pos, q), O.wolf_sum(R, pos, q, 0.3)]):
        assert abs(E.item() - r["E"]) <= TOL * 0.5 * np.abs(q * r["phi"]).sum()
        assert_atoms(F.cpu().numpy(), r["F"], TOL)
        assert_atoms(phi.cpu().numpy(), r["phi"], TOL)


# Two unit charges at distance d along x in one cell: the potential of the cutoff
# method is the kernel's 1 / sqrt(r2) of r2 = d^2 rounded, and nothing else.  Its
# steps are y = the seed (an FP32 number), t = x y rounded, r = 1 - t y, y + y r
# (1/2 + 3 r / 8) rounded: t's rounding moves the result by 2^-54 of itself, at
# most half an ulp, and the last rounding by half an ulp more.
@pytest.mark.parametrize("e", [-100, -31, -2, -1, 0, 1, 2, 30, 100])
def test_reciprocal_square_root(e, dev):
    from paper_1402_7216_gb300 import MSM
    unit = 2.0 ** e
    plan = MSM(box=4 * unit, periodic=False, cutoff=3 * unit, spacing=unit, order=3, splitting=2, precision="fp64",
               max_atoms=2)
    rng = np.random.default_rng(e + 200)
    edges = [1.0, 2.0, math.sqrt(2.0), math.sqrt(0.5), 0.5]  # where the mantissa or the exponent's parity of r2 turns over
    d = np.concatenate([rng.uniform(0.4, 2.99, 400), rng.uniform(0.999999, 1.000001, 50),
                        [np.nextafter(v, t) for v in edges for t in (0.0, v, 4.0)]]) * unit
    q = torch.ones(2, dtype=torch.float64, device=dev)
    P = torch.zeros((len(d), 2, 3), dtype=torch.float64, device=dev)
    P[:, 1, 0] = torch.tensor(d, device=dev)
    got = torch.stack([plan.cutoff_eval(p, q)[1][0] for p in P]).cpu().numpy()
    plan.check_status()
    with decimal.localcontext() as c:
        c.prec = 50
        for v, y in zip(d, got):
            err = abs(decimal.Decimal(float(y)) - 1 / decimal.Decimal(float(v) * float(v)).sqrt())
            assert err <= decimal.Decimal(math.ulp(float(y))) * decimal.Decimal("1.001"), (v, y)
