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
