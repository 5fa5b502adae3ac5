"""The in-place steps' FP64 collision: work it must not add to the pull step's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, FREESLIP, OUTFLOW, PRESSURE, VELOCITY, Case, to_gpu, with_random_state  # noqa: E402


@pytest.mark.parametrize("kinds", [None, (VELOCITY, OUTFLOW), (PRESSURE, FREESLIP)])
@pytest.mark.parametrize("lattice,n", [(D2Q9, (3, 3, 1)), (D2Q9, (33, 6, 1)), (D2Q9, (130, 7, 1)), (D3Q19, (3, 4, 3)),
                                       (D3Q19, (35, 5, 6))])
def test_in_place_steps_are_the_pull_steps_bit_for_bit(lattice, n, kinds):
    """Cells that update two to eight boundary nodes beside their own."""
    from paper_1710_02065_gb300 import lbm
    c = with_random_state(Case("aa", lattice, n, 0.57), seed=8, spread=0.05)
    spec = {VELOCITY: (VELOCITY, (0.04, 0.01, 0.0), None), OUTFLOW: (OUTFLOW, (0, 0, 0), None),
            PRESSURE: (PRESSURE, (0, 0, 0), None, 1.01), FREESLIP: (FREESLIP, (0, 0, 0), None)}
    for axis in range((2 if lattice == D2Q9 else 3) if kinds else 0):
        c.faces[2 * axis], c.faces[2 * axis + 1] = (spec[k] for k in (kinds if axis % 2 == 0 else kinds[::-1]))
        if n[axis] > 3:
            c.sponges[2 * axis + 1] = (2, 0.4)
    out = []
    for aa in (lbm.LBM_STREAM_PULL, lbm.LBM_STREAM_AA):
        s = to_gpu(c, 0)
        lbm.lbm_set_streaming(s.h, aa)
        s.step(4)
        out.append(s.populations())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


def test_a_large_in_place_step_costs_less_than_a_fifth_more_than_the_pull_step():
    """Both issue the same FP64 instructions per cell, which is what a 1024 x 1024
    step takes; with the collision's other routes in front of the target loop
    the in-place step issued 44 % more."""
    from paper_1710_02065_gb300 import lbm
    ms = []
    for aa in (lbm.LBM_STREAM_PULL, lbm.LBM_STREAM_AA):
        st = torch.cuda.Stream()
        s = lbm.Solver(D2Q9, (1024, 1024, 1), 0.6, lbm.LBM_FP64, stream=st.cuda_stream)
        lbm.lbm_set_streaming(s.h, aa)
        s.step(32)
        best = np.inf
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            s.step(32)
            e1.record(st)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
        s.close()
    assert ms[1] < 1.2 * ms[0], ms
