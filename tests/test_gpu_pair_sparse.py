"""GPU tests of the mixed pair kernel on plans whose cells hold few atoms (the
default capacity leaves cells of half a cutoff), on both sides of each line of
its dispatch: runs of atoms from 57,344 atoms on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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


# Cells and runs sum in different orders, so the bits tell which of the two the
# default took: runs leave most of the chip waiting below 57,344 atoms.
@pytest.mark.parametrize("cells,n,same", [(25, 5000, 2), (23, 57343, 2), (23, 57344, 1)], ids=str)
def test_default_takes_runs_by_atoms(cells, n, same, dev):
    box = 4.001 * cells
    pos, q = gas(n, box, seed=n)
    P = torch.tensor(pos, device=dev), torch.tensor(q, device=dev)
    F = {r: plan_of(box, True, pair_runs=r).cutoff_eval(*P)[2] for r in (0, 1, 2)}
    assert torch.equal(F[0], F[same]) and not torch.equal(F[0], F[3 - same])
