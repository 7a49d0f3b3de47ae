"""GPU tests of how the pair kernels hold their sums: contributions that
cancel, or that are far apart in size, must not cost the small ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


# Mixed plans of fewer than 2,048 cells share a group of targets among the four
# warps of a block; warp w takes every fourth step (64 sources of a neighbour
# row, 32 of the home cell) in the order of the input.  Here warp 0 meets
# sources of +2^18 and one small one, warp 1 sources of -2^18 and one small one,
# all at one distance: the large ones cancel exactly between the warps, and each
# small one is below half an ulp of its warp's total (2^23 or 2^22 against
# 0.19).  What remains is the small ones' sum, to the rounding of one pair: the
# distance is off by 4e-7 of itself at most (cell-local FP32 coordinates up to
# 10), the reciprocal square root by 2^-22.9.
@pytest.mark.parametrize("runs", [1, 2])
@pytest.mark.parametrize("step,x", [(32, 5.0), (64, 9.9)], ids=["home cell", "neighbour cell"])
def test_warps_join_their_totals_without_rounding(step, x, runs, dev):
    from paper_1402_7216_gb300 import MSM
    big, small, n = 2.0 ** 18, 0.375, 512
    q = np.zeros(n + 1)
    q[:step], q[step:2 * step] = big, -big
    q[4 * step], q[5 * step] = small, small
    q[n] = 1.0
    pos = np.full((n + 1, 3), 16.0)
    pos[:, 0] = x
    pos[n, 0] = x + 2.0  # the target, beyond the cells' border at 10.67 in the second case
    plan = MSM(box=32.0, periodic=False, cutoff=8.0, spacing=2.0, order=3, splitting=2, precision="mixed",
               max_atoms=n + 1, tuning=dict(pair_runs=runs))
    _, phi, F = plan.cutoff_eval(torch.tensor(pos, device=dev), torch.tensor(q, device=dev))
    torch.cuda.synchronize()
    plan.check_status()
    assert abs(phi[n].item() * 2.0 / (2 * small) - 1) <= 1e-6
    assert abs(F[n, 0].item() * 4.0 / (2 * small) - 1) <= 2e-6


# FP64 plans evaluate an MSM pair once, and add to the other atom's sums in
# memory.  A target between strong close charges (+2^47 at 0.5, -2^47 at 1.0: a
# potential of about 2^47, whose last bit is 2^-5) and 2,000 unit charges 5.5 to
# 7.8 away, each worth at most 0.011 there, under half that bit: added one by
# one onto the strong pairs' sum they vanish (their potential is about 8, some
# half of it by reactions).  The potential is linear in the charges, so the three
# evaluations may differ by a few last bits only (16 allowed: the sums a lane
# makes of 8 pairs and more before it adds them, the joins, the grid).  Which
# atom's group evaluates the strong pairs depends on the sorted order, hence
# several directions.
def test_far_pairs_survive_beside_close_ones(dev):
    from paper_1402_7216_gb300 import MSM
    n, big = 2000, 2.0 ** 47
    rng = np.random.default_rng(3)
    plan = MSM(box=24.0, periodic=False, cutoff=8.0, spacing=2.0, order=3, splitting=2, precision="fp64",
               max_atoms=n + 3)
    strong, weak = np.zeros(n + 3), np.ones(n + 3)
    strong[1:3] = big, -big
    weak[1:3] = 0.0
    Q = [torch.tensor(q, device=dev) for q in (strong + weak, strong, weak)]
    for _ in range(24):
        d = rng.normal(size=(n + 1, 3))
        d /= np.linalg.norm(d, axis=1)[:, None]
        near = np.outer([0.0, 0.5, -1.0], d[n])
        far = d[:n] * (rng.uniform(5.5 ** 3, 7.8 ** 3, n) ** (1 / 3))[:, None]
        P = torch.tensor(np.concatenate([near, far]) + 12.0, device=dev)
        both, s, w = (plan.eval(P, q)[1][0].item() for q in Q)
        assert 0.5 * big < s < 2 * big
        assert abs((both - s) - w) <= 16 * 2.0 ** -5
    plan.check_status()
