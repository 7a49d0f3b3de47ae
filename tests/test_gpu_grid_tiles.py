"""GPU tests of the per-level tiles of restriction and prolongation, the
real-input FFT passes and the FP64 stencil: the staged grids of FP64 plans
against the oracle's, on sizes around the tiles (4 coarse points, 32 x 8 x 8
and 32 x 4 x 4 fine points) and around 24^3 coarse points, where restriction
changes from tiles to axis passes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O

pytestmark = pytest.mark.gpu

# FP64 sums of at most a few thousand terms: 1e-13 of the largest value, two
# orders to spare (the bound of the FFT's staged grids elsewhere)
TOL = 1e-11


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("box,periodic,order,levels,method", [
    ((20.0, 24.0, 28.0), True, 3, 2, 2),      # 20 x 24 x 28 -> 10 x 12 x 14
    ((26.0, 18.0, 22.0), True, 5, 2, 1),      # 13 x 9 x 11 coarse points; stencil
    ((36.0, 20.0, 12.0), True, 5, 3, 2),      # 9 x 5 x 3 at the top
    ((48.0, 48.0, 48.0), True, 3, 2, 2),      # 24^3 coarse points: tiles
    ((50.0, 48.0, 48.0), True, 3, 2, 2),      # 25 x 24 x 24: axis passes
    ((70.0, 66.0, 64.0), True, 5, 2, 2),      # more than 64^3 fine points
    ((15.0, 22.0, 27.0), False, 3, 0, 0),
    ((13.0, 31.0, 16.0), False, 5, 3, 0),
])
def test_staged_grids_match_oracle(box, periodic, order, levels, method, dev):
    from paper_1402_7216_gb300 import MSM
    rng = np.random.default_rng(81)
    n, a = 400, 4.0
    pos, q = rng.uniform(0.0, 1.0, (n, 3)) * np.asarray(box), rng.uniform(-1.0, 1.0, n)
    plan = MSM(box=box, periodic=periodic, cutoff=a, spacing=1.0, levels=levels, order=order, splitting=2,
               precision="fp64", max_atoms=n, tuning=dict(lattice_method=method))
    P = O.Params(box=box, periodic=periodic, cutoff=a, spacing=1.0, levels=levels, order=order, split=2)
    ref = O.msm(P, pos, q, keep_grids=True)
    plan.eval(torch.tensor(pos, device=dev), torch.tensor(q, device=dev))
    plan.check_status()
    for k in range(plan.levels):
        for which, grids in (("q", ref["q_grids"]), ("u", ref["u_grids"])):
            got, want = plan.debug_grid(k, which), grids[k]
            assert np.abs(got - want).max() <= TOL * np.abs(want).max(), (k, which)
