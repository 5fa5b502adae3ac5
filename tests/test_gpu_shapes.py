"""Dispatch of the update kernels: the shapes and kernels lbm_step picks by
size, type and options against the explicitly chosen general kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, D3Q27, OUTFLOW, VELOCITY, Case, to_gpu, with_random_state  # noqa: E402

PRECS = {"fp64": 0, "fp32": 1, "fp16": 2, "bf16": 3}


def open_box(lattice, n, **kw):
    c = with_random_state(Case("shape", lattice, n, 0.6, **kw), seed=5, spread=0.02)
    c.faces = {0: (VELOCITY, (0.03, 0.0, 0.0), None), 1: (OUTFLOW, (0, 0, 0), None)}
    c.sponges = {1: (4, 0.4)}
    return c


def populations(c, prec, shape=None, steps=3):
    from paper_1710_02065_gb300 import lbm
    s = to_gpu(c, PRECS[prec])
    if shape:
        lbm.lbm_set_launch(s.h, *shape)
    got = lbm.lbm_get_launch(s.h)
    s.step(steps)
    lbm.lbm_sync(s.h)
    f = s.populations()
    s.close()
    return f, got


@pytest.mark.parametrize("nx,block", [(2, 32), (64, 32), (66, 64), (128, 64), (130, 96), (192, 96), (194, 64),
                                      (258, 32), (384, 64)])
@pytest.mark.parametrize("lattice", [D3Q19, D3Q27])
def test_default_block_leaves_no_idle_warp_and_changes_nothing(lattice, nx, block):
    """Rows of nx / 2 threads at the edges of the block rule: the reported
    default shape, and populations bitwise those of 64-thread blocks."""
    c = with_random_state(Case("shape", lattice, (nx, 4, 3), 0.6), seed=5, spread=0.02) if nx < 8 else \
        open_box(lattice, (nx, 4, 3))
    f, got = populations(c, "fp16")
    ref, _ = populations(c, "fp16", (64, 2))
    assert got == (block, 2)
    assert np.array_equal(f, ref)
