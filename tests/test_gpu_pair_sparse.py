"""GPU tests of the mixed pair kernel on plans whose cells hold few atoms (the
default capacity leaves cells of half a cutoff), on both sides of each line of
its dispatch: sources taken across ranges below 8 atoms a cell, a group shared by
four warps or not at 1,728 cells, runs of atoms from 57,344 atoms on.  Against
the oracle at the mixed path's tolerances (force rel-RMS 1e-5, potential 1e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from conftest import assert_atoms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def gas(n, box, seed):
    """n charges on a jittered lattice, at least 0.6 of its spacing apart."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1 / 3)))
    node = rng.permutation(m ** 3)[:n]
    ijk = np.stack([node % m, node // m % m, node // m ** 2], 1)
    return (ijk + 0.5 + rng.uniform(-0.2, 0.2, (n, 3))) * (box / m), rng.uniform(-1.0, 1.0, n)


def plan_of(box, periodic, **tuning):
    from paper_1402_7216_gb300 import MSM
    return MSM(box=box, periodic=periodic, cutoff=8.0, spacing=4.0, order=3, splitting=2, precision="mixed",
               tuning=tuning)  # the default capacity: cells of 4


@pytest.mark.parametrize("cells,n,periodic,runs", [
    (12, 8 * 1728 - 1, True, 0), (12, 8 * 1728, True, 0),    # across ranges or not
    (12, 18 * 1728 - 1, True, 0), (12, 18 * 1728, True, 0),  # a warp or four per group
    (11, 700, True, 0), (11, 8 * 1331, False, 0),            # four per group, nearly empty cells and full steps
    (13, 3001, False, 0), (7, 1500, True, 1), (13, 3001, True, 1), (13, 8 * 2197, False, 1),
], ids=str)
def test_sparse_cells_match_oracle(cells, n, periodic, runs, dev):
    box = 4.001 * cells
    pos, q = gas(n, box, seed=cells + n)
    plan = plan_of(box, periodic, pair_runs=runs)
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    E, phi, F = plan.eval(*P)
    again = plan.eval(*P)
    wolf = plan.wolf_eval(*P, 0.3)
    plan.check_status()
    par = O.Params(box=(box,) * 3, periodic=periodic, cutoff=8.0, spacing=4.0, order=3, split=2)
    ref, wref = O.msm(par, pos, q), O.wolf_sum(par, pos, q, 0.3)
    assert_atoms(F.cpu().numpy(), ref["F"], 1e-5)
    assert_atoms(phi.cpu().numpy(), ref["phi"], 1e-6)
    assert_atoms(wolf[2].cpu().numpy(), wref["F"], 1e-5)
    assert torch.equal(F, again[2]) and torch.equal(phi, again[1])


# Cells and runs sum in different orders, so the bits tell which of the two the
# default took: below 16,384 cells runs leave most of the chip waiting unless there
# are 57,344 atoms.
@pytest.mark.parametrize("cells,n,same", [(25, 5000, 2), (23, 57343, 2), (23, 57344, 1), (26, 5000, 1)], ids=str)
def test_default_takes_runs_by_atoms(cells, n, same, dev):
    box = 4.001 * cells
    pos, q = gas(n, min(box, 92.0), seed=n)  # dense enough for sums whose order shows
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    F = {r: plan_of(box, True, pair_runs=r).cutoff_eval(*P)[2] for r in (0, 1, 2)}
    assert torch.equal(F[0], F[same]) and not torch.equal(F[0], F[3 - same])


def test_batch_of_sparse_replicas(dev):
    """A batch graph takes the same walks (a group is never shared there)."""
    from paper_1402_7216_gb300 import MSMBatch
    boxes, counts = (60.0, 45.0, 70.0), (4000, 2500, 9000)
    systems = [gas(n, b, seed=n) for n, b in zip(counts, boxes)]
    pos = torch.tensor(np.concatenate([p for p, _ in systems]), device=dev)
    q = torch.tensor(np.concatenate([c for _, c in systems]), device=dev)
    E, phi, F = torch.empty(3, dtype=torch.float64, device=dev), torch.empty_like(q), torch.empty_like(pos)
    batch = MSMBatch([plan_of(b, True) for b in boxes])
    batch.graph(pos, q, list(counts), E, phi, F).launch()
    torch.cuda.synchronize()
    o = 0
    for (p, c), b in zip(systems, boxes):
        ref = O.msm(O.Params(box=(b,) * 3, periodic=True, cutoff=8.0, spacing=4.0, order=3, split=2), p, c)
        assert_atoms(F[o:o + len(c)].cpu().numpy(), ref["F"], 1e-5)
        assert_atoms(phi[o:o + len(c)].cpu().numpy(), ref["phi"], 1e-6)
        o += len(c)
