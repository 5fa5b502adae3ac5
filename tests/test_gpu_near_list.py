"""The list of cells next to a solid that a geometry upload builds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [(3, 3, 1), (5, 5, 1), (9, 7, 1), (17, 8, 1), (8, 4, 1)])
def test_force_with_one_solid_at_every_place(n):
    """Cell counts that are and are not a multiple of eight, a solid at each of
    the first and last cells: the force of the links of every other cell."""
    from paper_1710_02065_gb300 import lbm
    N = n[0] * n[1]
    rng = np.random.default_rng(1)
    s = lbm.Solver(0, n, 0.7, lbm.LBM_FP64)
    _, _, xi, w = lbm.lbm_lattice_table(0)
    f = w[:, None] * (1 + 0.1 * rng.standard_normal((9, N)))
    s.set_populations(f)
    for at in sorted({*range(min(N, 12)), *range(max(0, N - 12), N)}):
        solid = np.zeros(N, np.uint8)
        solid[at] = 1
        lbm.lbm_set_geometry(s.h, solid)
        F = np.zeros(3)
        for c in range(N):
            x, y = c % n[0], c // n[0]
            for i in range(1, 9):
                if c != at and (x + xi[i][0]) % n[0] + n[0] * ((y + xi[i][1]) % n[1]) == at:
                    F[:2] += 2 * xi[i][:2] * f[i, c]
        assert np.abs(lbm.lbm_force(s.h, 0) - F).max() < 1e-14, at
    s.close()
