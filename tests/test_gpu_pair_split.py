"""GPU tests of the mixed pair kernel's group shapes: cells or runs of atoms
per warp, on both sides of 2,048 cells (below, a block's four warps share a
group's sources), with ranges of sources that end inside a step of 64, wrap
around a periodic row, or hold nothing, against the oracle.  Tolerances: those
of the mixed path everywhere (force rel-RMS 1e-5, potential 1e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from conftest import assert_atoms
from synth import make_water_box

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("runs", [1, 2])
@pytest.mark.parametrize("box,waters,periodic,cutoff,fill", [
    ((50.0, 46.0, 53.0), 2000, True, 6.0, 1),   # ~1.5 atoms per cell: short and empty ranges
    ((42.0, 38.0, 45.0), 1900, True, 6.0, 12),   # 7 cells along x
    ((40.0, 45.0, 38.0), 1500, False, 6.0, 1),
    ((40.0, 45.0, 38.0), 1500, False, 9.0, 40),  # more than 32 atoms per cell
])
def test_group_shapes_match_oracle(box, waters, periodic, cutoff, fill, runs, dev):
    from paper_1402_7216_gb300 import MSM
    pos, q = make_water_box(box, waters, 3, 3, seed=71, periodic=periodic)
    plan = MSM(box=box, periodic=periodic, cutoff=cutoff, spacing=2.0, order=3, splitting=2, precision="mixed",
               max_atoms=len(q), tuning=dict(cell_fill=fill, pair_runs=runs))
    ref = O.msm(O.Params(box=box, periodic=periodic, cutoff=cutoff, spacing=2.0, order=3, split=2), pos, q)
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    E, phi, F = plan.eval(*P)
    again = plan.eval(*P)
    torch.cuda.synchronize()
    plan.check_status()
    assert abs(E.item() - ref["E"]) <= 1e-6 * abs(ref["E"])
    assert_atoms(F.cpu().numpy(), ref["F"], 1e-5)
    assert_atoms(phi.cpu().numpy(), ref["phi"], 1e-6)
    assert torch.equal(F, again[2]) and torch.equal(phi, again[1])
