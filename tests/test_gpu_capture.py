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
