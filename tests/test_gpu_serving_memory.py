"""Host memory of the solve server's requests."""
import ctypes

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


def _mixed(lend, aa):
    """Results of six requests of both lattices on a server that lends `lend` bytes."""
    from paper_1710_02065_gb300 import lbm
    s = lbm.lbm_server_create(1 << 28, 4)
    lbm.lbm_server_set_host_memory(s, lend, 1 << 20)
    if aa:
        lbm.lbm_server_set_streaming(s, lbm.LBM_STREAM_AA)
    ids, sizes = [], []
    for k in range(6):
        lattice, n = ((0, (64 + k, 40, 1)), (1, (18, 9 + k, 11)))[k % 2]
        rho, u = _state(n, k)
        if k == 2:
            rho = None
        if k == 3:
            u = None
        ids.append(lbm.lbm_server_submit(s, lattice, k % 3, n, 0.7, 3 + 4 * k, rho, u))
        sizes.append(int(np.prod(n)))
    out = _collect(s, ids, sizes)
    lbm.lbm_server_destroy(s)
    return out


@pytest.mark.parametrize("aa", [False, True])
def test_pageable_requests_give_the_page_locked_ones_results(aa):
    """No page-locked memory lent, some of it, all of it: the same bits."""
    ref = _mixed(1 << 30, aa)
    for lend in (0, 200000):
        for (r0, u0), (r1, u1) in zip(ref, _mixed(lend, aa)):
            assert np.isfinite(r0).all() and np.array_equal(r0, r1) and np.array_equal(u0, u1)


class _PoolProps(ctypes.Structure):
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locationType", ctypes.c_int),
                ("locationId", ctypes.c_int), ("win32", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


def test_request_without_device_memory_for_its_upload_stays_queued():
    """A pageable request whose lattice fits and whose staging buffer does not
    (the device's memory pool is bounded to lie between): it waits with its
    state and is served once memory is there."""
    from paper_1710_02065_gb300 import lbm
    n = (4096, 2048, 1)  # in place, 16 bits: lattice 151 MB, staging 268 MB
    N = 4096 * 2048
    rng = np.random.default_rng(0)
    rho = 1 + 0.01 * rng.standard_normal(N)
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    props = _PoolProps(allocType=1, locationType=1, maxSize=320 << 20)
    pool, old = ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(old), torch.cuda.current_device()) == 0
    out = []
    for bounded in (True, False):
        s = lbm.lbm_server_create(8 << 30, 2)
        lbm.lbm_server_set_streaming(s, lbm.LBM_STREAM_AA)
        lbm.lbm_server_set_host_memory(s, 0, 0)
        rid = lbm.lbm_server_submit(s, 0, lbm.LBM_FP16_SHIFTED, n, 0.7, 3, rho)
        if bounded:
            assert cu.cuDeviceSetMemPool(torch.cuda.current_device(), pool) == 0
            try:
                for _ in range(2):
                    lbm.lbm_server_run(s, 4)
                    assert lbm.lbm_server_poll(s, rid) == (lbm.LBM_REQ_QUEUED, 0)
            finally:
                assert cu.cuDeviceSetMemPool(torch.cuda.current_device(), old) == 0
        out.append(_collect(s, [rid], [N])[0])
        lbm.lbm_server_destroy(s)
    torch.cuda.synchronize()
    assert cu.cuMemPoolDestroy(pool) == 0
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


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
