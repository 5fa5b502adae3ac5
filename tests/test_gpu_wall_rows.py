"""D2Q9 rows on walls and other faces of the y axis in the vectorised kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, FREESLIP, OUTFLOW, PRESSURE, VELOCITY, Case, to_gpu, with_random_state  # noqa: E402

PRECS = {"fp64": 0, "fp32": 1, "fp16": 2, "bf16": 3}


def spec(kind, face, n):
    rng = np.random.default_rng(face)
    prof = 0.03 * rng.standard_normal((n[1] if face < 2 else n[0], 3))
    prof[:, 2] = 0
    return {VELOCITY: (VELOCITY, (0, 0, 0), prof), OUTFLOW: (OUTFLOW, (0, 0, 0), None),
            PRESSURE: (PRESSURE, (0, 0, 0), None, 1.01), FREESLIP: (FREESLIP, (0, 0, 0), None)}[kind]


@pytest.mark.parametrize("nx,ny", [(4, 3), (6, 4), (64, 5), (66, 3), (130, 6)])
@pytest.mark.parametrize("xkinds", [None, (VELOCITY, OUTFLOW), (OUTFLOW, PRESSURE), (FREESLIP, VELOCITY)])
@pytest.mark.parametrize("ykinds", [(FREESLIP, FREESLIP), (VELOCITY, PRESSURE), (PRESSURE, OUTFLOW), (OUTFLOW, VELOCITY)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
def test_face_rows_against_the_general_kernel(prec, ykinds, xkinds, nx, ny):
    """Every face rule on the y axis, corners with every rule of the x axis,
    sponge layers and inlet noise: two cells per thread against one.  FP64 bit
    for bit; FP32: 1e-5 of the largest deviation from the mean; 16-bit storage:
    one rounding of each stored value per step and the start (2^-10, 2^-7 of the
    largest)."""
    from paper_1710_02065_gb300 import lbm
    n = (nx, ny, 1)
    c = with_random_state(Case("rows", D2Q9, n, 0.6), seed=9, spread=0.05)
    for axis, kinds in enumerate((xkinds, ykinds)):
        for side in range(2 if kinds else 0):
            c.faces[2 * axis + side] = spec(kinds[side], 2 * axis + side, n)
    c.noise = (4, 0.01)
    if ny > 4:
        c.sponges = {2: (2, 0.3)}
        if xkinds and nx > 6:
            c.sponges[1] = (3, 0.4)
    out = []
    for cells in (1, 2):
        s = to_gpu(c, PRECS[prec])
        lbm.lbm_set_launch(s.h, 0, cells)
        assert lbm.lbm_get_launch(s.h)[1] == cells
        s.step(3)
        lbm.lbm_sync(s.h)
        out.append(s.populations())
        s.close()
    assert np.isfinite(out[0]).all()
    if prec == "fp64":
        assert np.array_equal(out[0], out[1])
    else:
        dev = np.abs(out[0] - out[0].mean(axis=1, keepdims=True)).max()
        tol = {"fp32": 1e-5, "fp16": 4 * 2.0 ** -10, "bf16": 4 * 2.0 ** -7}[prec]
        assert np.abs(out[1] - out[0]).max() <= tol * dev


def step_us(n, prec, kinds, aa, cells):
    from paper_1710_02065_gb300 import lbm
    st = torch.cuda.Stream()
    s = lbm.Solver(D2Q9, n, 0.6, PRECS[prec], stream=st.cuda_stream)
    for face, kind in enumerate(kinds):
        lbm.lbm_set_boundary(s.h, face, kind, (0.03, 0.0, 0.0) if kind == VELOCITY else None)
    if aa:
        lbm.lbm_set_streaming(s.h, lbm.LBM_STREAM_AA)
    lbm.lbm_set_launch(s.h, 0, cells)
    s.step(320)
    best = np.inf
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        s.step(320)
        e1.record(st)
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) / 320 * 1e3)
    s.close()
    return best


@pytest.mark.parametrize("n", [(128, 128, 1), (400, 200, 1)])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_default_shape_between_walls_is_not_the_slower_one(prec, n):
    """Free-slip walls, pull: the default against one cell per thread, with a
    quarter for timing and the edges' longer code (it was 1.2 to 1.45 times)."""
    kinds = (VELOCITY, OUTFLOW, FREESLIP, FREESLIP)
    assert step_us(n, prec, kinds, False, 0) < 1.25 * step_us(n, prec, kinds, False, 1)


@pytest.mark.parametrize("prec,n,cells", [("fp32", (600, 600, 1), 1), ("fp32", (600, 602, 1), 2), ("fp16", (600, 350, 1), 1),
                                          ("bf16", (600, 352, 1), 2), ("fp32", (64, 6, 1), 1)])
@pytest.mark.parametrize("walls", [True, False])
def test_small_in_place_lattices_take_one_cell_per_thread(prec, n, cells, walls):
    """At the edges of the rule; a periodic y axis keeps two, as does the pull."""
    from paper_1710_02065_gb300 import lbm
    s = lbm.Solver(D2Q9, n, 0.6, PRECS[prec])
    for face in (2, 3) if walls else ():
        lbm.lbm_set_boundary(s.h, face, FREESLIP)
    assert lbm.lbm_get_launch(s.h)[1] == 2
    lbm.lbm_set_streaming(s.h, lbm.LBM_STREAM_AA)
    assert lbm.lbm_get_launch(s.h)[1] == (cells if walls else 2)
    lbm.lbm_set_launch(s.h, 0, 2)
    assert lbm.lbm_get_launch(s.h)[1] == 2
    s.close()


@pytest.mark.parametrize("n", [(128, 128, 1), (400, 200, 1)])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_default_in_place_shape_is_not_the_slower_one(prec, n):
    """The default against one cell per thread, with a tenth for timing (it was
    1.2 to 1.35 times)."""
    kinds = (VELOCITY, OUTFLOW, OUTFLOW, OUTFLOW)
    assert step_us(n, prec, kinds, True, 0) < 1.1 * step_us(n, prec, kinds, True, 1)
