"""GPU tests of the FP64 pair sums that evaluate a pair once for both atoms:
neighbours in one group and in different groups of targets, across the periodic
boundary, and sums cleared from one evaluation to the next on one plan (more
and fewer atoms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from conftest import assert_atoms

pytestmark = pytest.mark.gpu

# sums of ~1,000 FP64 terms, each rounded to 2^-53: 1e-13 of the RMS, two
# orders to spare
TOL = 1e-11


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n", [2, 8, 9, 33, 257, 1300])
def test_pairs_once_for_both_atoms(n, periodic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_7216_gb300 import MSM
    dev = torch.device("cuda:0")
    box = np.array([30.0, 28.0, 26.0])
    rng = np.random.default_rng(n)
    pos, q = rng.uniform(0.0, 1.0, (n, 3)) * box, rng.uniform(-1.0, 1.0, n)
    corner = rng.uniform(-4.0, 4.0, (n - n // 2, 3))  # half of them around one corner
    pos[n // 2:] = np.mod(corner, box) if periodic else np.abs(corner)
    par = dict(box=tuple(box), periodic=periodic, cutoff=8.0, spacing=2.0, order=3)
    plan = MSM(splitting=2, precision="fp64", max_atoms=n, **par)
    P = O.Params(split=2, **par)
    for m in (n, n - n // 3, n):
        E, phi, F = plan.eval(torch.tensor(pos[:m], device=dev), torch.tensor(q[:m], device=dev))
        plan.check_status()
        ref = O.msm(P, pos[:m], q[:m])
        assert abs(E.item() - ref["E"]) <= TOL * 0.5 * np.abs(q[:m] * ref["phi"]).sum() + 1e-300
        assert_atoms(F.cpu().numpy(), ref["F"], TOL)
        assert_atoms(phi.cpu().numpy(), ref["phi"], TOL)


@pytest.mark.parametrize("n", [19440, 19441, 65536])
def test_groups_of_8_and_16(n):
    """Both sides of the change of targets per group, and a size well above."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_7216_gb300 import MSM
    dev = torch.device("cuda:0")
    box = np.array([88.0, 86.0, 90.0]) * (n / 65536) ** (1 / 3)
    rng = np.random.default_rng(n)
    pos, q = rng.uniform(0.0, 1.0, (n, 3)) * box, rng.uniform(-1.0, 1.0, n)
    par = dict(box=tuple(box), periodic=True, cutoff=8.0, spacing=3.0, order=3)
    E, phi, F = MSM(splitting=2, precision="fp64", max_atoms=n, **par).eval(torch.tensor(pos, device=dev),
                                                                            torch.tensor(q, device=dev))
    ref = O.msm(O.Params(split=2, **par), pos, q)
    assert abs(E.item() - ref["E"]) <= TOL * 0.5 * np.abs(q * ref["phi"]).sum()
    assert_atoms(F.cpu().numpy(), ref["F"], TOL)
    assert_atoms(phi.cpu().numpy(), ref["phi"], TOL)
