"""Calls made while the caller captures a CUDA graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_captured_steps_replay_as_direct_ones(precision):
    """Single steps captured by the caller, replayed: bit for bit the same
    number of direct steps."""
    from paper_1710_02065_gb300 import lbm
    rng = np.random.default_rng(2)
    rho, u = 1 + 0.01 * rng.standard_normal(96 * 50), 0.02 * rng.standard_normal((96 * 50, 3))
    u[:, 2] = 0
    out = []
    for captured in (True, False):
        st = torch.cuda.Stream()
        s = lbm.Solver(0, (96, 50, 1), 0.7, precision, stream=st.cuda_stream)
        s.set_state(rho, u)
        lbm.lbm_sync(s.h)
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                lbm.lbm_step(s.h, 1)
                lbm.lbm_step(s.h, 1)
            with torch.cuda.stream(st):
                for _ in range(5):
                    g.replay()
        else:
            s.step(10)
        lbm.lbm_sync(s.h)
        out.append(s.populations())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("before,after", [("disc", "many"), ("many", "disc"), ("none", "disc"), ("disc", "none")])
def test_captured_force_follows_the_geometry(level, before, after):
    """A captured force sample replayed after the cell types changed (longer,
    shorter, empty lists of cells next to a solid): the direct call's bits."""
    from paper_1710_02065_gb300 import lbm
    st = torch.cuda.Stream()
    s = lbm.Solver(0, (96, 64, 1), 0.7, lbm.LBM_FP32, stream=st.cuda_stream)
    n = (96, 64)
    if level:
        lbm.lbm_add_refinement_patch(s.h, (20, 16, 0), (40, 30, 0))
        n = (81, 61)
    x, y = np.meshgrid(np.arange(n[0]), np.arange(n[1]))
    masks = {"disc": (x - 40) ** 2 + (y - 30) ** 2 < 60, "many": (x % 3 == 0) & (y % 2 == 0) & (x > 2) & (y > 2),
             "none": np.zeros_like(x)}
    rng = np.random.default_rng(2)
    u = 0.02 * rng.standard_normal((x.size, 3))
    u[:, 2] = 0
    lbm.lbm_set_geometry_level(s.h, level, masks[before].astype(np.uint8).reshape(-1))
    lbm.lbm_set_state_level(s.h, level, 1 + 0.01 * rng.standard_normal(x.size), u)
    lbm.lbm_sync(s.h)
    F = torch.full((3,), 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        lbm.lbm_force_async(s.h, level, F.data_ptr())
    for which in (before, after):
        lbm.lbm_set_geometry_level(s.h, level, masks[which].astype(np.uint8).reshape(-1))
        with torch.cuda.stream(st):
            g.replay()
        lbm.lbm_sync(s.h)
        direct = lbm.lbm_force(s.h, level)
        assert np.array_equal(F.cpu().numpy(), direct) and direct.any() == (which != "none")
    s.close()
