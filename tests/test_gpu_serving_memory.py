"""Host memory of the solve server's requests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _state(n, seed):
    rng = np.random.default_rng(seed)
    N = int(np.prod(n))
    u = 0.02 * rng.standard_normal((N, 3))
    if n[2] == 1:
        u[:, 2] = 0
    return 1 + 0.01 * rng.standard_normal(N), u


def _collect(s, ids, sizes, steps=7):
    from paper_1710_02065_gb300 import lbm
    out = {}
    for _ in range(1000):
        lbm.lbm_server_run(s, steps)
        for rid, N in zip(ids, sizes):
            if rid not in out and lbm.lbm_server_poll(s, rid)[0] in (lbm.LBM_REQ_DONE, lbm.LBM_REQ_FAILED):
                rho, u = np.empty(N), np.empty((N, 3))
                assert lbm.lbm_server_result(s, rid, rho, u) == lbm.LBM_OK
                out[rid] = (rho, u)
        if len(out) == len(ids):
            break
    return [out[rid] for rid in ids]


def test_submit_while_the_caller_captures_a_graph():
    """A submit between the caller's captured launches neither fails nor ends
    the capture, and its request is served."""
    from paper_1710_02065_gb300 import lbm
    n = (64, 48, 1)
    rho, u = _state(n, 1)
    s = lbm.lbm_server_create(1 << 28, 8)
    x = torch.zeros(16, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        x += 1
        ids = [lbm.lbm_server_submit(s, 0, lbm.LBM_FP32, n, 0.7, 20, rho, u)]
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert (x == 2).all()
    ids.append(lbm.lbm_server_submit(s, 0, lbm.LBM_FP32, n, 0.7, 20, rho, u))
    a, b = _collect(s, ids, [64 * 48] * 2)
    lbm.lbm_server_destroy(s)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
