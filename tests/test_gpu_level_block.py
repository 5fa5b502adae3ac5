"""lbm_set_launch's block size on refined 2D levels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("ext", [(4, 4), (5, 4), (33, 20)])
def test_block_size_changes_nothing(ext, precision):
    """Every block size reaches the substep kernel of both refined levels, whose
    roles end inside blocks of each: bit for bit the default's populations."""
    from paper_1710_02065_gb300 import lbm
    rng = np.random.default_rng(3)
    out = []
    for block in (0, 32, 96, 128, 256):
        s = lbm.Solver(0, (60, 40, 1), 0.6, precision)
        lbm.lbm_add_refinement_patch(s.h, (4, 5, 0), (*ext, 0))
        n = [2 * e + 1 for e in ext]
        levels = 2
        if n[0] > 12:
            lbm.lbm_add_refinement_patch(s.h, (6, 4, 0), (9, 7, 0))
            levels = 3
            solid = np.zeros((n[1], n[0]), np.uint8)
            solid[-6, -8:-5] = 1
            lbm.lbm_set_geometry_level(s.h, 1, solid.reshape(-1))
        lbm.lbm_set_launch(s.h, block, 1)
        rng = np.random.default_rng(3)
        for level in range(levels):
            e, _ = lbm.lbm_level_info(s.h, level)
            N = int(np.prod(e))
            u = 0.02 * rng.standard_normal((N, 3))
            u[:, 2] = 0
            lbm.lbm_set_state_level(s.h, level, 1 + 0.01 * rng.standard_normal(N), u)
        s.step(5)
        lbm.lbm_sync(s.h)
        f = []
        for level in range(levels):
            e, _ = lbm.lbm_level_info(s.h, level)
            a = np.zeros((9, int(np.prod(e))))
            lbm.lbm_get_populations_level(s.h, level, a)
            f.append(a)
        out.append(f)
        s.close()
    for f in out[1:]:
        assert all(np.isfinite(a).all() and np.array_equal(a, b) for a, b in zip(out[0], f))
