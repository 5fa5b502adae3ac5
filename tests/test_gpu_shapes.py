"""Dispatch of the update kernels: the shapes and kernels lbm_step picks by
size, type and options against the explicitly chosen general kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, D3Q27, FREESLIP, OUTFLOW, PRESSURE, VELOCITY, Case, to_gpu, with_random_state  # noqa: E402

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


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("ext", [(4, 4), (5, 4), (4, 33), (67, 5)])
def test_level_step_2d_on_small_and_long_patches(ext, prec, tol):
    """The refined level's substep with its coupling at the smallest ring, odd
    extents and long sides (rings that end inside a block of every role),
    against the oracle; both levels after three coarse steps."""
    import oracle
    from cases import to_oracle
    from paper_1710_02065_gb300 import inputs, lbm
    n, patch = (80, 44, 1), (3, 4, *ext)
    nf = (2 * ext[0] + 1, 2 * ext[1] + 1)
    c = Case("patch", D2Q9, n, 0.6)
    c.rho0, c.u0 = inputs.uniform_flow_perturbed(n[0], n[1], 0.05, 4, rel=0.2)
    rho_f, u_f = inputs.uniform_flow_perturbed(*nf, 0.05, 5, rel=0.2)
    P, _ = to_oracle(c)
    T = oracle.TwoLevel(P, *patch)
    T.init(c.rho0, c.u0, rho_f, u_f)
    s = to_gpu(c, PRECS[prec])
    lbm.lbm_add_refinement_patch(s.h, (*patch[:2], 0), (*ext, 1))
    lbm.lbm_set_state_level(s.h, 1, rho_f, u_f)
    lbm.lbm_set_state(s.h, c.rho0, c.u0)
    T.run(3)
    s.step(3)
    live = np.ones((n[1], n[0]), bool)
    live[patch[1] + 2:patch[1] + ext[1] - 1, patch[0] + 2:patch[0] + ext[0] - 1] = False  # frozen covered cells
    for level, (Q, f, keep) in enumerate(((T.Pc, T.fc, live.reshape(-1)), (T.Pf, T.ff, slice(None)))):
        r, u, _ = Q.moments(f)
        gr, gu = np.zeros(Q.ncell), np.zeros((Q.ncell, 3))
        lbm.lbm_moments_level(s.h, level, gr, gu, None)
        assert np.linalg.norm((gr - r)[keep]) <= tol * np.linalg.norm(r[keep])
        assert np.linalg.norm((gu - u)[keep]) <= tol * np.linalg.norm(u[keep])
    s.close()


@pytest.mark.parametrize("lattice,n,solids", [(D2Q9, (9, 9, 1), "cell"), (D2Q9, (40, 9, 1), "wall"),
                                              (D3Q19, (9, 8, 7), "cell"), (D3Q27, (160, 130, 5), "wall")])
def test_force_sums_every_link(lattice, n, solids):
    """Lists of fewer cells than a block, not a whole number of blocks, and
    more than one turn of the largest grid (41,600 cells next to a wall);
    twice in a row, so that the block counter is seen to be back at zero.  The
    sums have at most 1.9 M terms of magnitude < 0.6: 1e-10 absolute covers
    their FP64 round-off.  The reference is the exact sum over the links (the
    oracle adds them one after the other, which alone loses 1e-10 here)."""
    import math
    import oracle
    from cases import to_oracle
    from paper_1710_02065_gb300 import lbm
    c = with_random_state(Case("force", lattice, n, 0.6), seed=6, spread=0.3)
    m = np.zeros((n[2], n[1], n[0]), np.uint8)
    if solids == "cell":
        m[n[2] // 2, 4, 4] = 1
    else:
        m[n[2] // 2, n[1] // 2 if lattice == D2Q9 else slice(None), :] = 1
    c.solid = m.reshape(-1)
    P, f = to_oracle(c)
    _, q, xi, _, _ = oracle.lattice(lattice)
    sums = [math.fsum(f[i].reshape(m.shape)[(np.roll(m, -xi[i][::-1], (0, 1, 2)) == 1) & (m == 0)]) for i in range(q)]
    ref = np.array([math.fsum(2.0 * xi[i][a] * sums[i] for i in range(q)) for a in range(3)])
    assert np.abs(P.wall_force(f) - ref).max() < 1e-8
    s = to_gpu(c, PRECS["fp64"])
    for _ in range(2):
        assert np.abs(lbm.lbm_force(s.h, 0) - ref).max() < 1e-10
    dev = torch.full((3,), 7.0, dtype=torch.float64, device="cuda")
    lbm.lbm_force_async(s.h, 0, dev.data_ptr())
    lbm.lbm_sync(s.h)
    assert np.abs(dev.cpu().numpy() - ref).max() < 1e-10
    lbm.lbm_set_geometry(s.h, None)
    assert not lbm.lbm_force(s.h, 0).any()
    s.close()


@pytest.mark.parametrize("rho_ref", [1.0, 1.02])
@pytest.mark.parametrize("kinds", [(VELOCITY, OUTFLOW), (PRESSURE, FREESLIP), (FREESLIP, PRESSURE)])
@pytest.mark.parametrize("lattice,n", [(D2Q9, (3, 9, 1)), (D2Q9, (33, 5, 1)), (D2Q9, (65, 7, 1)), (D3Q19, (3, 4, 5)),
                                       (D3Q19, (31, 4, 5)), (D3Q19, (34, 5, 4))])
def test_fp64_collision_form(lattice, n, kinds, rho_ref):
    """Warps of bulk, sponge and face cells together (rows of 3 to 65 cells),
    every face rule on every axis, rest and other sponge references, against
    the oracle: populations (order 0.1) to 1e-13 after three steps, some
    hundred roundings of 1.1e-16 each."""
    from cases import to_oracle
    c = with_random_state(Case("fp64", lattice, n, 0.57), seed=8, spread=0.05)
    spec = {VELOCITY: (VELOCITY, (0.04, 0.01, 0.0), None), OUTFLOW: (OUTFLOW, (0, 0, 0), None),
            PRESSURE: (PRESSURE, (0, 0, 0), None, 1.01), FREESLIP: (FREESLIP, (0, 0, 0), None)}
    for axis in range(2 if lattice == D2Q9 else 3):
        c.faces[2 * axis], c.faces[2 * axis + 1] = (spec[k] for k in (kinds if axis % 2 == 0 else kinds[::-1]))
        c.sponges[2 * axis + 1] = (2, 0.4)
    c.rho_ref = rho_ref
    c.noise = (4, 0.01)
    P, f = to_oracle(c)
    f = P.run(f, 3)
    got, _ = populations(c, "fp64")
    assert np.abs(got - f).max() < 1e-13


@pytest.mark.parametrize("nx", [4, 6, 34, 62, 66, 130])
@pytest.mark.parametrize("faces", ["periodic", "open x", "outflow y", "free-slip y"])
@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("lattice,prec", [(D2Q9, "fp32"), (D2Q9, "fp16"), (D2Q9, "bf16"), (D3Q19, "fp16"),
                                          (D3Q27, "bf16")])
def test_vector_rows_and_shift_against_the_general_kernel(lattice, prec, shift, faces, nx):
    """The rows the 2D vector path takes (wrapped, outflow faces), the ones it
    leaves, and the storage shift in the vector kernel: default shape against
    one cell per thread.  FP32: 1e-5 of the largest deviation from the mean;
    16-bit storage: one rounding of each stored value per step and the start
    (2^-10, 2^-7 of the largest)."""
    from paper_1710_02065_gb300 import lbm
    n = (nx, 7, 1) if lattice == D2Q9 else (nx, 6, 5)
    c = with_random_state(Case("rows", lattice, n, 0.6), seed=9, spread=0.05)
    if faces == "open x":
        c.faces = {0: (VELOCITY, (0.03, 0.0, 0.0), None), 1: (OUTFLOW, (0, 0, 0), None)}
        c.sponges = {1: (2, 0.4)}
    elif faces != "periodic":
        kind = OUTFLOW if faces == "outflow y" else FREESLIP
        c.faces = {2: (OUTFLOW, (0, 0, 0), None), 3: (kind, (0, 0, 0), None)}
        c.sponges = {2: (3, 0.3)}
    out = []
    for shape in ((128, 1), None):
        s = to_gpu(c, PRECS[prec])
        if shift:
            lbm.lbm_set_storage_shift(s.h, (0.05, 0.02, 0.0))
        if shape:
            lbm.lbm_set_launch(s.h, *shape)
        assert lbm.lbm_get_launch(s.h)[1] == (1 if shape else 2)
        s.step(3)
        lbm.lbm_sync(s.h)
        out.append(s.populations())
        s.close()
    dev = np.abs(out[0] - out[0].mean(axis=1, keepdims=True)).max()
    tol = {"fp32": 1e-5, "fp16": 4 * 2.0 ** -10, "bf16": 4 * 2.0 ** -7}[prec]
    assert np.abs(out[1] - out[0]).max() <= tol * dev


@pytest.mark.parametrize("option", ["order 4", "sponge reference", "solid", "odd row"])
def test_options_the_vector_kernel_leaves_run_the_general_one(option):
    from paper_1710_02065_gb300 import lbm
    c = open_box(D2Q9, (33 if option == "odd row" else 34, 7, 1))
    if option == "sponge reference":
        c.u_ref = (0.03, 0.0, 0.0)
    if option == "solid":
        c.solid = np.eye(1, c.ncell, 50, dtype=np.uint8)[0]
    s = to_gpu(c, PRECS["fp32"])
    if option == "order 4":
        lbm.lbm_set_hermite_order(s.h, 4)
    assert lbm.lbm_get_launch(s.h) == (128, 1)
    s.close()


@pytest.mark.parametrize("noise", [0.0, 0.01])
@pytest.mark.parametrize("lattice,prec,n", [(D2Q9, "fp64", (16, 16, 1)), (D2Q9, "fp16", (256, 250, 1)),
                                            (D2Q9, "fp32", (512, 640, 1)), (D3Q19, "fp32", (33, 40, 39)),
                                            (D3Q19, "bf16", (160, 64, 60)), (D3Q27, "fp16", (64, 48, 40))])
def test_chained_launches_are_the_plain_ones_bit_for_bit(lattice, prec, n, noise):
    """Steps on a stream of their own run as chained launches (captured pairs
    without inlet noise, single launches with it; lattices below and above the
    early-start size), on the legacy stream as plain ones."""
    from paper_1710_02065_gb300 import lbm
    c = open_box(lattice, n)
    out = []
    for stream in (0, torch.cuda.Stream().cuda_stream):
        s = lbm.Solver(c.lattice, c.n, c.tau, PRECS[prec], stream=stream)
        for face, spec in c.faces.items():
            lbm.lbm_set_boundary(s.h, face, *spec)
        for face, (w, chi) in c.sponges.items():
            lbm.lbm_set_sponge(s.h, face, w, chi)
        lbm.lbm_set_inlet_noise(s.h, 3, noise)
        s.set_populations(c.f0)
        s.step(67)
        s.step(3)
        lbm.lbm_sync(s.h)
        out.append(s.populations())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


@pytest.mark.parametrize("lattice,prec,n,shape,aa", [
    (D3Q27, "fp16", (192, 128, 128), (128, 1), False), (D3Q19, "fp32", (129, 128, 128), None, False),
    (D3Q19, "bf16", (256, 160, 192), (128, 1), True), (D2Q9, "fp32", (2048, 2100, 1), None, False),
    (D2Q9, "fp16", (2048, 4200, 1), None, True)])
def test_sweep_direction_changes_nothing(lattice, prec, n, shape, aa):
    """Lattices beyond twice the L2 sweep every other step backwards: a field
    with the period of a box of 1/8 the cells or less (swept forwards) stays
    that box's, bit for bit, at even and odd step counts."""
    from paper_1710_02065_gb300 import lbm
    small = tuple(max(1, e // 4) if a else e for a, e in enumerate(n))
    rng = np.random.default_rng(3)
    out = []
    rho0 = 1 + 0.01 * rng.standard_normal(small[::-1])
    u0 = 0.02 * rng.standard_normal(small[::-1] + (3,))
    if lattice == D2Q9:
        u0[..., 2] = 0
    for m in (small, n):
        reps = tuple(b // a for a, b in zip(small, m))[::-1]
        s = lbm.Solver(lattice, m, 0.7, PRECS[prec])
        if aa:
            lbm.lbm_set_streaming(s.h, lbm.LBM_STREAM_AA)
        if shape:
            lbm.lbm_set_launch(s.h, *shape)
        s.set_state(np.tile(rho0, reps).reshape(-1), np.tile(u0, reps + (1,)).reshape(-1, 3))
        got = []
        for steps in (4, 1):
            s.step(steps)
            rho = np.empty(int(np.prod(m)), np.float32)
            u = np.empty((rho.size, 3), np.float32)
            lbm.lbm_moments_f32(s.h, rho, u)
            got.append((rho.reshape(m[::-1]), u.reshape(m[::-1] + (3,))))
        out.append((got, reps))
        s.close()
    (a, _), (b, reps) = out
    for (r0, v0), (r1, v1) in zip(a, b):
        assert np.array_equal(np.tile(r0, reps), r1) and np.array_equal(np.tile(v0, reps + (1,)), v1)
