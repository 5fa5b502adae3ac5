"""FP64 densities beyond the range of single precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from cases import D2Q9, D3Q19, OUTFLOW, PRESSURE, VELOCITY, Case, to_gpu, to_oracle  # noqa: E402


@pytest.mark.parametrize("cells", [1, 2])
@pytest.mark.parametrize("faces", ["periodic", "velocity", "pressure"])
@pytest.mark.parametrize("scale", [1e-3, 1e3, 1e37, 1e39, 1e150])
@pytest.mark.parametrize("lattice,n", [(D2Q9, (36, 8, 1)), (D3Q19, (20, 6, 5))])
def test_fp64_step_scales_with_the_density(lattice, n, scale, faces, cells):
    """Two steps of a field of density `scale` (1 + 1 % variation): bulk cells,
    velocity and constant-density nodes, both kernels, against the oracle:
    1e-12 of the largest population."""
    from paper_1710_02065_gb300 import lbm
    rng = np.random.default_rng(4)
    N = int(np.prod(n))
    u = 0.03 * rng.standard_normal((N, 3))
    if lattice == D2Q9:
        u[:, 2] = 0
    c = Case("range", lattice, n, 0.7, rho0=scale * (1 + 0.01 * rng.standard_normal(N)), u0=u)
    if faces == "velocity":
        c.faces = {0: (VELOCITY, (0.03, 0.01, 0.0), None), 1: (OUTFLOW, (0, 0, 0), None)}
    elif faces == "pressure":
        c.faces = {0: (OUTFLOW, (0, 0, 0), None), 1: (PRESSURE, (0, 0, 0), None, scale)}
    P, f = to_oracle(c)
    f = P.run(f, 2)
    s = to_gpu(c, 0)
    lbm.lbm_set_launch(s.h, 0, cells)
    s.step(2)
    got = s.populations()
    s.close()
    assert np.abs(got - f).max() <= 1e-12 * np.abs(f).max()


@pytest.mark.parametrize("n", [(36, 8, 1), (35, 8, 1), (20, 6, 5)])
def test_fp64_served_step_scales_with_the_density(n):
    """The solve server's update (two cells per lane, one on odd rows) at 1e39."""
    import oracle
    from paper_1710_02065_gb300 import lbm
    rng = np.random.default_rng(4)
    lattice, N = (D2Q9 if n[2] == 1 else D3Q19), int(np.prod(n))
    u0 = 0.03 * rng.standard_normal((N, 3))
    if lattice == D2Q9:
        u0[:, 2] = 0
    rho0 = 1e39 * (1 + 0.01 * rng.standard_normal(N))
    P = oracle.Problem(lattice, n, 0.7)
    rho, u, _ = P.moments(P.run(P.equilibrium(rho0, u0), 2))
    s = lbm.lbm_server_create(1 << 28, 2)
    rid = lbm.lbm_server_submit(s, lattice, 0, n, 0.7, 2, rho0, u0)
    lbm.lbm_server_run(s, 2)
    r, v = np.empty(N), np.empty((N, 3))
    lbm.lbm_server_result(s, rid, r, v)
    lbm.lbm_server_destroy(s)
    assert np.abs(r - rho).max() <= 1e-12 * rho.max() and np.abs(v - u).max() <= 1e-12


PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "rr.cuh"
__global__ void k(int n, const double *x, double *r, double *q)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    r[t] = rr::recip_fma(x[t]);
    q[t] = 1.0 / x[t];
}
int main(int argc, char **argv)
{
    FILE *f = fopen(argv[1], "rb");
    const int n = atoi(argv[2]);
    std::vector<double> x(n), r(2 * n);
    if (fread(x.data(), 8, n, f) != (size_t)n) return 1;
    fclose(f);
    double *xd, *rd;
    if (cudaMalloc(&xd, 8 * n) != cudaSuccess || cudaMalloc(&rd, 16 * n) != cudaSuccess) return 2;
    cudaMemcpy(xd, x.data(), 8 * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(n, xd, rd, rd + n);
    if (cudaMemcpy(r.data(), rd, 16 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    f = fopen(argv[1], "wb");
    fwrite(r.data(), 8, 2 * n, f);
    fclose(f);
    return 0;
}
"""


def test_reciprocal_over_the_whole_range(tmp_path):
    """recip_fma against the quotient: one unit in the last place (half of one
    each from the rounding of the two) for normal x below 2^1022; infinity for 0
    and subnormal x, 0 for the rest."""
    import subprocess
    from paper_1710_02065_gb300 import build
    rng = np.random.default_rng(6)
    edge = [2.0 ** k * (1 + s * 2.0 ** -52) for k in (-1021, -127, -1, 0, 1, 127, 1021) for s in (-1, 0, 1)]
    x = np.concatenate([1 + 0.2 * rng.standard_normal(200000), 2.0 ** rng.uniform(-1021, 1021, 200000), np.array(edge),
                        [0.0, 5e-324, 1e-310, 1e-46, 3.4e38, 3.5e38, 1.7e308, np.inf, np.nan]])
    x = np.concatenate([x, -x])
    src, exe, data = tmp_path / "recip.cu", tmp_path / "recip", tmp_path / "x.bin"
    src.write_text(PROGRAM)
    x.tofile(data)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", str(exe),
                    str(src)], check=True)
    subprocess.run([str(exe), str(data), str(x.size)], check=True)
    r, q = np.fromfile(data).reshape(2, -1)
    normal = (np.abs(x) >= 2.0 ** -1022) & (np.abs(x) < 2.0 ** 1022)
    assert (np.abs(r[normal] - q[normal]) <= np.spacing(np.abs(q[normal]))).all()
    tiny = np.abs(x) < 2.0 ** -1022
    assert np.array_equal(r[tiny], np.copysign(np.inf, x[tiny])) and not r[~normal & ~tiny].any()
