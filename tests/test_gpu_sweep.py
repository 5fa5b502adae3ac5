"""The backward sweep: taken where the rule says, and changing nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, D3Q27  # noqa: E402

Q = {D2Q9: 9, D3Q19: 19, D3Q27: 27}
ELEM = (8, 4, 2, 2)


def planes_beyond_twice_the_l2(lattice, prec, cells):
    """The number of planes (rows in 2D) of `cells` cells beyond which a step
    moves more than twice the bytes of this device's L2."""
    l2 = torch.cuda.get_device_properties(torch.cuda.current_device()).L2_cache_size
    return 2 * l2 // (2 * Q[lattice] * ELEM[prec] * cells)


@pytest.mark.parametrize("noise", [0.0, 0.01])
@pytest.mark.parametrize("lattice,prec,plane,shape,aa", [
    (D2Q9, 1, (1024,), None, False), (D2Q9, 2, (1024,), None, True), (D2Q9, 0, (1023,), (128, 1), False),
    (D3Q19, 1, (128, 64), None, False), (D3Q19, 1, (129, 64), None, False), (D3Q19, 3, (128, 128), (128, 1), False),
    (D3Q19, 2, (128, 64), (128, 1), True), (D3Q19, 2, (129, 64), None, True), (D3Q27, 2, (96, 64), None, False)])
def test_sweep_alternates_beyond_twice_the_l2_and_changes_nothing(lattice, prec, plane, shape, aa, noise):
    """One plane below the line every step sweeps forwards; twice beyond it every
    other one backwards (single launches with inlet noise set, captured pairs
    without), and a field with the period of the small box stays that box's.
    (D3Q19 with one cell per thread: the vectorised kernel leaves the small box's
    wrapped planes to the general update, which rounds differently.)"""
    from paper_1710_02065_gb300 import lbm
    last = planes_beyond_twice_the_l2(lattice, prec, int(np.prod(plane)))
    rng = np.random.default_rng(3)
    small = plane + (last,)
    shape3 = (small + (1,) if lattice == D2Q9 else small)
    rho0 = 1 + 0.01 * rng.standard_normal(shape3[::-1])
    u0 = 0.02 * rng.standard_normal(shape3[::-1] + (3,))
    if lattice == D2Q9:
        u0[..., 2] = 0
    axis = 1 if lattice == D2Q9 else 0  # of the arrays: the last axis of the lattice
    got = []
    for reps in (1, 2):
        n = list(shape3)
        n[1 if lattice == D2Q9 else 2] *= reps
        s = lbm.Solver(lattice, n, 0.7, prec, stream=torch.cuda.Stream().cuda_stream)
        if aa:
            lbm.lbm_set_streaming(s.h, lbm.LBM_STREAM_AA)
        if shape:
            lbm.lbm_set_launch(s.h, *shape)
        if noise:
            lbm.lbm_set_inlet_noise(s.h, 1, noise)  # (no inlet: no effect but on the launches)
        tile = [1, 1, 1]
        tile[axis] = reps
        s.set_state(np.tile(rho0, tile).reshape(-1), np.tile(u0, tile + [1]).reshape(-1, 3))
        seen, fields = [], []
        for steps in (1, 1, 2, 1):
            seen.append(lbm.lbm_get_sweep(s.h))
            s.step(steps)
        rho = np.empty(int(np.prod(n)), np.float32)
        u = np.empty((rho.size, 3), np.float32)
        lbm.lbm_moments_f32(s.h, rho, u)
        s.close()
        assert sorted(set(seen)) == ([False] if reps == 1 else [False, True]), seen
        if reps == 2:
            assert seen[0] != seen[1] and seen[1] != seen[2] and seen[2] == seen[3]
        fields = [np.split(a.reshape(tuple(n[::-1]) + a.shape[1:]), reps, axis=axis) for a in (rho, u)]
        got.append(fields)
    for small_field, large in zip(*got):
        for part in large:
            assert np.array_equal(small_field[0], part)
