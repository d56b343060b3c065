"""GPU tests of the explicit kernels at the edges of their tiles, copies and
z-chunks: two steps with a flow that changes sign, against the oracle."""
import numpy as np
import pytest

from oracle import ch_oracle as co
from paper_2105_01865_gb300 import inputs

from _parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

P, N, D = co.PERIODIC, co.NOFLUX, co.DIRICHLET


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2105_01865_gb300 import build, capi
    build.build()
    capi.load()


# (nz, ny, nx): one cell short of, at and past the tile, the smallest box, several z-chunks
@pytest.mark.parametrize("shape", [(5, 5, 5), (17, 9, 31), (16, 8, 32), (15, 7, 33), (33, 17, 65), (6, 24, 64)])
@pytest.mark.parametrize("bc", [(P, P, P), (P, N, N), (N, P, D)])
@pytest.mark.parametrize("flow", [True, False])
def test_two_steps_match_oracle(shape, bc, flow):
    from paper_2105_01865_gb300.solver import Solver
    nz, ny, nx = shape
    h, cn, pe = 1.0 / 16, 0.75 / 16, 20.0
    rng = np.random.default_rng(nx * ny)
    C0 = 0.5 + 0.4 * rng.standard_normal(shape)  # sharp everywhere: every WENO weight differs
    vel = None
    if flow:
        vel = inputs.curl_velocity(*(inputs.uniform_faces(n, n * h) for n in (nx, ny, nz)), bc, seed=nx, kmax=3)
    s = Solver(shape, h, bc, cn, pe, 0.2 * h, C0, precision="f64", advect=flow)
    if flow:
        s.set_velocity_fine(*vel)
    s.step(2)
    got = s.field()
    H3, H2 = s.explicit_terms()
    s.close()
    p = co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=0.2 * h, bc=bc)
    ref = co.step(C0, vel, p, 2)
    # the bar of the other FP64 tests; rounding alone gives about 1e-15
    assert_parity(got, ref, 1e-12, f"FP64 explicit {shape} {bc} flow={flow}")


# the FP32 kernel's copies: whole 16-byte chunks (nx a multiple of 4; walls
# reverse the last one), element by element otherwise, a lone last column
@pytest.mark.parametrize("nx", [5, 8, 12, 63, 64, 65, 66, 68, 129])
@pytest.mark.parametrize("bc", [(P, P, P), (N, P, N), (N, N, D)])
@pytest.mark.parametrize("flow", [True, False])
def test_fp32_two_steps_match_oracle(nx, bc, flow):
    from paper_2105_01865_gb300.solver import Solver
    nz, ny = 9, 17
    shape = (nz, ny, nx)
    h, cn, pe = 1.0 / 16, 0.75 / 16, 20.0
    rng = np.random.default_rng(nx)
    C0 = (0.5 + 0.4 * rng.standard_normal(shape)).astype(np.float32).astype(np.float64)
    vel = None
    if flow:
        vel = inputs.curl_velocity(*(inputs.uniform_faces(n, n * h) for n in (nx, ny, nz)), bc, seed=nx, kmax=3)
        vel = [a.astype(np.float32).astype(np.float64) for a in vel]
    s = Solver(shape, h, bc, cn, pe, 0.2 * h, C0, precision="f32", advect=flow)
    if flow:
        s.set_velocity_fine(*vel)
    s.step(2)
    got = s.field()
    s.close()
    ref = co.step(C0, vel, co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=0.2 * h, bc=bc), 2)
    # the bar of the other FP32 tests of a few steps
    assert_parity(got, ref, 1e-6, f"FP32 explicit {shape} {bc} flow={flow}")


DIV_PROBE = """
#include "ch_explicit64.cuh"
__global__ void div_kernel(const double* a, const double* b, double* q, long n) {
    const long i = blockIdx.x * 256L + threadIdx.x;
    if (i < n) q[i] = chg::div_newton(a[i], b[i]);
}
extern "C" int div_probe(const double* a, const double* b, double* q, long n) {
    div_kernel<<<(unsigned)((n + 255) / 256), 256>>>(a, b, q, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_weno_quotient_is_a_division(tmp_path):
    """The FP64 WENO5 quotient over every exponent a sum of weights can have: within a unit in the last
    place of a / b, and the same as a / b where b or its reciprocal is near the subnormals, or not a number."""
    import ctypes
    import subprocess
    from paper_2105_01865_gb300 import build
    src, lib = tmp_path / "div.cu", tmp_path / "libdiv.so"
    src.write_text(DIV_PROBE)
    subprocess.run(["nvcc", *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)], check=True)
    rng = np.random.default_rng(1)
    with np.errstate(all="ignore"):
        e = np.concatenate([rng.uniform(-1074, 1023, 200_000), np.repeat([-1074, -1023, -1022, -801, -800, -799, 999, 1000,
                                                                         1001, 1022, 1023], 2000).astype(float)])
        b = np.ldexp(rng.uniform(1, 2, e.size), e.astype(int))
        g = np.ldexp(rng.uniform(-2, 2, e.size), rng.integers(-60, 1, e.size))  # the quotient: differences of C
        a = b * g
        edge = np.array([0.0, -0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, 1.0])
        a, b = np.append(a, np.repeat(edge, edge.size)), np.append(b, np.tile(edge, edge.size))
        ref = a / b
    ta, tb = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
    tq = torch.empty_like(ta)
    fn = ctypes.CDLL(str(lib)).div_probe
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_long]
    torch.cuda.synchronize()
    assert fn(ta.data_ptr(), tb.data_ptr(), tq.data_ptr(), ta.numel()) == 0
    q = tq.cpu().numpy()
    near = (b >= 2.0 ** -799) & (b < 2.0 ** 1000)
    assert np.array_equal(q[~near & (b < 2.0 ** -800)], ref[~near & (b < 2.0 ** -800)], equal_nan=True)
    assert np.array_equal(q[b >= 2.0 ** 1001], ref[b >= 2.0 ** 1001], equal_nan=True)
    assert np.array_equal(q[np.isnan(b)], ref[np.isnan(b)], equal_nan=True)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(q), fin)
    ulps = np.abs(q[fin] - ref[fin]) / np.spacing(np.abs(ref[fin]))
    print(f"quotient: at most {ulps.max():.0f} units in the last place from a / b, {np.mean(ulps > 0):.1e} of them not equal")
    assert ulps.max() <= 1


# a regulariser whose fourth power is subnormal or zero in the weights of a constant region
@pytest.mark.parametrize("weno_eps", [1e-6, 1e-79, 1e-80])
def test_fp64_small_regulariser(weno_eps):
    from paper_2105_01865_gb300.solver import Solver
    shape, bc, h, cn, pe = (9, 12, 40), (P, N, N), 1.0 / 16, 0.75 / 16, 20.0
    C0 = np.zeros(shape)
    C0[:, :, 12:20] = 1.0  # constant on both sides
    vel = inputs.curl_velocity(*(inputs.uniform_faces(n, n * h) for n in shape[::-1]), bc, seed=5, kmax=3)
    s = Solver(shape, h, bc, cn, pe, 0.2 * h, C0, precision="f64", weno_eps=weno_eps, advect=True)
    s.set_velocity_fine(*vel)
    s.step(1)
    got = s.field()
    s.close()
    nz, ny, nx = shape
    p = co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=0.2 * h, bc=bc, eps=weno_eps)
    assert_parity(got, co.step(C0, vel, p, 1), 1e-12, f"weno_eps {weno_eps}")


def depth_fp32(nx, ny, nz, slots):
    """Planes a FP32 tile marches (explicit_depth in ch_step.cu): the depth whose waves take the least."""
    xy, best = -(-nx // 64) * -(-ny // 8), None
    for c in range(1, nz + 1):
        tz = -(-nz // c)
        cost = -(-(xy * -(-nz // tz)) // slots) * (tz + 2.0)
        if best is None or cost < best[0]:
            best = (cost, tz)
    return best[1]


# rows of any kind, even rows, aligned rows with walls and without; tiles of several planes, the last one shorter
@pytest.mark.parametrize("nx", [67, 66, 68])
@pytest.mark.parametrize("bc", [(P, P, P), (N, P, P), (N, N, N), (P, P, N), (P, N, D), (N, P, D)])
@pytest.mark.parametrize("flow", [True, False])
def test_fp32_deep_tiles_match_oracle(nx, bc, flow):
    from paper_2105_01865_gb300.solver import Solver
    nz, ny = 11, 597
    for slots in (2 * 152, 3 * 152):
        tz = depth_fp32(nx, ny, nz, slots)
        assert tz >= 3 and nz % tz != 0
    h, cn, pe = 1.0 / 16, 0.75 / 16, 20.0
    rng = np.random.default_rng(nx)
    C0 = (0.5 + 0.4 * rng.standard_normal((nz, ny, nx))).astype(np.float32).astype(np.float64)
    vel = None
    if flow:
        vel = inputs.curl_velocity(*(inputs.uniform_faces(n, n * h) for n in (nx, ny, nz)), bc, seed=nx, kmax=3)
        vel = [a.astype(np.float32).astype(np.float64) for a in vel]
    s = Solver((nz, ny, nx), h, bc, cn, pe, 0.2 * h, C0, precision="f32", advect=flow)
    if flow:
        s.set_velocity_fine(*vel)
    s.step(1)
    got = s.field()
    s.close()
    ref = co.step(C0, vel, co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=0.2 * h, bc=bc), 1)
    # the bar of the other FP32 tests of a few steps
    assert_parity(got, ref, 1e-6, f"FP32 deep tiles nx={nx} {bc} flow={flow}")
