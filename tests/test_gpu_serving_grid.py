"""The batched update's grid: fewer warps per SM on large groups."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _rate(lattice, prec, n, count, aa, launch):
    """Cell updates per second (device time, best of three rounds)."""
    from paper_1710_02065_gb300 import lbm
    s = lbm.lbm_server_create(16 << 30, 16)
    if aa:
        lbm.lbm_server_set_streaming(s, lbm.LBM_STREAM_AA)
    lbm.lbm_server_set_launch(s, lattice, prec, *launch)
    for _ in range(count):
        lbm.lbm_server_submit(s, lattice, prec, n, 0.6, 1 << 40)
    lbm.lbm_server_run(s, 20)
    best = np.inf
    for _ in range(3):
        t0 = lbm.lbm_server_gpu_time(s)
        lbm.lbm_server_run(s, 20)
        best = min(best, lbm.lbm_server_gpu_time(s) - t0)
    lbm.lbm_server_destroy(s)
    return count * int(np.prod(n)) * 20 / (best * 1e-3)


@pytest.mark.parametrize("n,count", [((128, 128, 128), 4), ((160, 160, 160), 1)])
def test_default_shape_of_a_large_fp32_group_is_the_faster_one(n, count):
    """D3Q19 FP32 beyond the L2: two cells per lane, the default, against one, with
    2 % for the timing."""
    assert _rate(1, 1, n, count, False, (0, 0)) > 0.98 * _rate(1, 1, n, count, False, (1, 4))


@pytest.mark.parametrize("lattice,prec,n,count,aa", [(1, 1, (96, 96, 96), 3, False), (1, 1, (66, 130, 140), 2, False),
                                                     (1, 1, (64, 64, 64), 2, False), (1, 2, (100, 90, 80), 2, True)])
def test_result_does_not_depend_on_the_grid(lattice, prec, n, count, aa):
    """Groups with and without the bound, tiles filled in part: bit for bit the
    one-cell shape, whose grid has none."""
    from paper_1710_02065_gb300 import lbm
    N = int(np.prod(n))
    rng = np.random.default_rng(5)
    rho, u = 1 + 0.01 * rng.standard_normal(N), 0.02 * rng.standard_normal((N, 3))
    out = []
    for launch in ((0, 0), (1, 4)):
        s = lbm.lbm_server_create(16 << 30, 16)
        if aa:
            lbm.lbm_server_set_streaming(s, lbm.LBM_STREAM_AA)
        lbm.lbm_server_set_launch(s, lattice, prec, *launch)
        ids = [lbm.lbm_server_submit(s, lattice, prec, n, 0.7, 4 + k, rho, u) for k in range(count)]
        lbm.lbm_server_run(s, 8)
        for rid in ids:
            r, v = np.empty(N), np.empty((N, 3))
            assert lbm.lbm_server_result(s, rid, r, v) == lbm.LBM_OK
            out.append((r, v))
        lbm.lbm_server_destroy(s)
    for (r0, v0), (r1, v1) in zip(out[:count], out[count:]):
        assert np.isfinite(r0).all() and np.array_equal(r0, r1) and np.array_equal(v0, v1)
