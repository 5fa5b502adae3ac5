"""lbm_get_launch reports the shape the next lbm_step runs, for any handle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, OUTFLOW, VELOCITY  # noqa: E402


@pytest.mark.parametrize("n,faces", [((34, 7, 1), [(0, VELOCITY)]), ((34, 2, 1), [(2, OUTFLOW), (3, OUTFLOW)])])
def test_answers_before_the_handle_is_configured(n, faces):
    """One face of an axis set so far, or an axis too short for its faces:
    lbm_step refuses, the query answers."""
    from paper_1710_02065_gb300 import lbm
    s = lbm.Solver(D2Q9, n, 0.6, lbm.LBM_FP32)
    for face, kind in faces:
        lbm.lbm_set_boundary(s.h, face, kind, (0.0, 0.0, 0.0))
    assert lbm.lbm_get_launch(s.h) == (32, 2)
    with pytest.raises(lbm.LBMError):
        s.step(1)
    s.close()


@pytest.mark.parametrize("vec,block,got", [(2, 0, (128, 1)), (2, 64, (64, 1)), (0, 0, (128, 1))])
@pytest.mark.parametrize("option", ["bgk", "order 4", "sponge reference", "radial sponge", "storage shift", "solid"])
def test_reports_the_general_kernel_where_it_runs(option, vec, block, got):
    """Options the vectorised kernel does not take, with an explicit and with
    the default shape."""
    from paper_1710_02065_gb300 import lbm
    shifted = option == "storage shift"
    n = (34, 6, 5) if shifted else (34, 7, 1)
    s = lbm.Solver(D3Q19 if shifted else D2Q9, n, 0.6, lbm.LBM_FP32)
    lbm.lbm_set_launch(s.h, block, vec)
    if vec and option not in ("storage shift", "solid"):
        pytest.skip("an explicit shape is reported whatever collision and sponges are selected")
    if vec:
        assert lbm.lbm_get_launch(s.h)[1] == vec
    if option == "bgk":
        lbm.lbm_set_collision(s.h, 1)
    elif option == "order 4":
        lbm.lbm_set_hermite_order(s.h, 4)
    elif option == "sponge reference":
        lbm.lbm_set_boundary(s.h, 0, VELOCITY, (0.03, 0.0, 0.0))
        lbm.lbm_set_boundary(s.h, 1, OUTFLOW)
        lbm.lbm_set_sponge(s.h, 1, 4, 0.4, 1.0, (0.03, 0.0, 0.0))
    elif option == "radial sponge":
        lbm.lbm_set_radial_sponge(s.h, (17.0, 3.0, 0.0), 1.0, 4.0, 0.3)
    elif shifted:
        lbm.lbm_set_storage_shift(s.h, (0.05, 0.0, 0.0))
    else:
        lbm.lbm_set_geometry(s.h, np.eye(1, s.ncell, 50, dtype=np.uint8)[0])
    assert lbm.lbm_get_launch(s.h) == got
    s.close()
