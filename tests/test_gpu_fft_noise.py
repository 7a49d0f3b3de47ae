"""GPU test of the FP32 transforms' rounding noise in the lattice cutoff.

Charges sit on the level-0 grid points (h = 2 exactly), so the charge grid is
exact and the mixed plan's potential grid differs from the FP64 plan's by the
transforms' rounding alone.  The charges are random numbers minus the mean of
their six neighbours, strong in the short waves and weak in the long ones that
make the potential, as neutral molecules are.  In a float32 model of the passes,
complex transforms of the whole grid leave 1.6e-6 (48^3) and 1.7e-6 (80^3) of
the potential's RMS, transforms of two real rows at once without smoothing
2.2e-6 and 2.3e-6, and with it 1.4e-6 and 1.5e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [48, 80])
def test_mixed_potential_grid_noise(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_7216_gb300 import MSM
    dev = torch.device("cuda:0")
    g = np.random.default_rng(n).uniform(-1.0, 1.0, (n, n, n))
    q = g - sum(np.roll(g, s, ax) for s in (1, -1) for ax in range(3)) / 6.0
    q = np.round(q * 2.0 ** 20) / 2.0 ** 20
    z, y, x = np.meshgrid(*[2.0 * np.arange(n)] * 3, indexing="ij")
    P = torch.tensor(np.stack([x, y, z], 3).reshape(-1, 3), device=dev)
    Q = torch.tensor(q.reshape(-1), device=dev)
    u = {}
    for precision in ("fp64", "mixed"):
        plan = MSM(box=2.0 * n, periodic=True, cutoff=10.0, spacing=2.0, order=3, splitting=2, precision=precision,
                   max_atoms=n ** 3)
        assert plan.dims[0] == (n, n, n) and plan.lattice_method == "fft"
        plan.eval(P, Q)
        assert np.array_equal(np.asarray(plan.debug_grid(0, "q")), q)
        u[precision] = np.asarray(plan.debug_grid(0, "u"))
        plan.check_status()
    d = u["mixed"] - u["fp64"]
    assert np.sqrt((d ** 2).mean()) <= 1.85e-6 * np.sqrt((u["fp64"] ** 2).mean())
