"""GPU tests of the line solvers: one u = 0 step against the oracle where blocks,
restarts and ghost rows can go wrong (line lengths about the block sizes, lines
shorter than the restart distance, every wall type, every copy width), for
operators of each restart distance and for one that decays too slowly and takes
the scan solvers; and on boxes with lines enough for the streaming form."""
import numpy as np
import pytest

from oracle import ch_oracle as co
from paper_2105_01865_gb300 import inputs

import _line_form as lf
from _parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

P, N, D = co.PERIODIC, co.NOFLUX, co.DIRICHLET
# (nz, ny, nx): lines of 5 to 3 blocks and a remainder; nx odd, even, a multiple of 4
SHAPES = [(5, 6, 7), (31, 33, 32), (64, 65, 34), (33, 5, 97), (100, 31, 66), (7, 129, 36), (129, 8, 5), (6, 40, 160)]
BCS = [(P, P, P), (N, N, N), (P, N, D), (N, P, P)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2105_01865_gb300 import build, capi
    build.build()
    capi.load()


# boxes with more than 304 groups of 32 lines (1216 where rows are not 16-byte
# aligned): the directions that stream, with a partial last block and last group
STREAMED = [((104, 96, 72), "f32"),    # x, y
            ((66, 100, 100), "f32"),   # z
            ((200, 200, 67), "f32"),   # x unaligned
            ((200, 70, 197), "f32"),   # y unaligned
            ((70, 199, 197), "f32"),   # z unaligned
            ((98, 100, 520), "f64")]   # x in FP64, too long for a tile


@pytest.mark.parametrize("shape, prec", STREAMED)
@pytest.mark.parametrize("bc", [(P, P, P), (N, N, D)])
@pytest.mark.parametrize("ck", [0.25, 12.0])
def test_streamed_lines_match_oracle(shape, prec, bc, ck):
    test_one_step_matches_oracle(shape, ck, prec, bc)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("shape", SHAPES)
# ck of the first substep: restart distances of 1, 2 and 3 blocks, and the scan solvers
@pytest.mark.parametrize("ck", [0.02, 1.2, 12.0, 400.0])
def test_one_step_matches_oracle(shape, ck, prec, bc=None):
    from paper_2105_01865_gb300.solver import Solver
    nz, ny, nx = shape
    h, cn, pe = 1.0 / 32, 0.75 / 32, 100.0
    bc = bc or BCS[(SHAPES.index(shape) + int(ck)) % len(BCS)]
    dt = ck / (8.0 / 15.0 / pe / 2.0 * 4.0 * cn ** 2 / h ** 4)
    rng = np.random.default_rng(nx)
    C0 = inputs.drops_field(shape, h, bc, [(nx * h / 2, ny * h / 3, nz * h / 2)], [0.3 * min(shape) * h], cn)
    C0 = C0 + 0.05 * rng.standard_normal(shape)
    if prec == "f32":
        C0 = C0.astype(np.float32).astype(np.float64)
    s = Solver(shape, h, bc, cn, pe, dt, C0, precision=prec)
    s.step(1)
    got = s.field()
    s.close()
    ref = co.step(C0, None, co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=dt, bc=bc), 1)
    # backward-stable solves: a few roundings times the condition number of (I + ck [1,-4,6,-4,1])
    assert_parity(got, ref, 8 * (1 + 16 * ck) * 2.0 ** (-53 if prec == "f64" else -24), f"march {shape} {bc} ck={ck} {prec}")


# boxes that take every form of the line solvers in every direction, copy width and kind of wall
# (test_march_factors.py counts them)
@pytest.mark.parametrize("shape, prec, ck", lf.BOXES)
@pytest.mark.parametrize("bc", [(P, P, P), (N, N, D)])
def test_every_form_matches_oracle(shape, prec, ck, bc):
    test_one_step_matches_oracle(shape, ck, prec, bc)


# FP32 boxes too large for the oracle: rows of single-element copies, and over 6080 groups of 64 columns, the last
# one partial, which take two columns a thread; restarts of one block of 32 rows and of three
@pytest.mark.parametrize("shape, ck", [((501, 501, 501), 0.25), ((130, 620, 628), 0.25), ((130, 620, 628), 12.0),
                                       ((1020, 200, 324), 0.25), ((1020, 200, 324), 12.0)])
@pytest.mark.parametrize("bc", [(P, P, P), (P, N, N), (N, P, D)])
def test_large_boxes_match_fp64(shape, bc, ck):
    """One step against the library's FP64 form, which the oracle pins above."""
    from paper_2105_01865_gb300.solver import Solver
    assert lf.forms("f32", bc, shape, ck).count("march") >= (3 if ck < 1 else 2)
    h, cn, pe = 1.0 / 32, 0.75 / 32, 100.0
    dt = ck / (8.0 / 15.0 / pe / 2.0 * 4.0 * cn ** 2 / h ** 4)
    gen = torch.Generator(device="cuda").manual_seed(shape[0])
    C0 = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    out = {}
    for prec in ("f64", "f32"):
        s = Solver(shape, h, bc, cn, pe, dt, C0, precision=prec)
        s.step(1)
        s.sync()
        out[prec] = s.C.double()
        s.close()
    d = out["f32"] - out["f64"]
    l2, em = float(d.norm() / out["f64"].norm()), float(d.abs().max() / out["f64"].abs().max())
    bar = 8 * (1 + 16 * ck) * 2.0 ** -24  # as above
    print(f"{shape} {bc} ck={ck}: rel L2 {l2:.2e}, max elem {em:.2e} (bar {bar:.1e})")
    assert l2 <= bar and em <= 10 * bar


# an operator that decays too slowly to restart, on a smooth field (whose small differences FP32 keeps): the
# scan and column solvers of 65- to 256-row lines, even and odd rows, which other boxes of these sizes no longer take
# (FP64 also with Dirichlet walls, next to which such a field changes by more than itself)
@pytest.mark.parametrize("shape", [(90, 100, 66), (150, 200, 34), (66, 250, 72), (70, 130, 67)])
@pytest.mark.parametrize("prec, bc", [("f64", (P, P, P)), ("f64", (P, P, N)), ("f64", (N, N, D)), ("f32", (P, P, P)),
                                      ("f32", (P, P, N))])
def test_scan_solvers_match_oracle(shape, bc, prec):
    from paper_2105_01865_gb300.solver import Solver
    ck = 60.0
    assert lf.forms(prec, bc, shape, ck) == ("scan",) * 3
    nz, ny, nx = shape
    h, cn, pe = 1.0 / 32, 0.75 / 32, 1e4
    dt = ck / (8.0 / 15.0 / pe / 2.0 * 4.0 * cn ** 2 / h ** 4)
    x, y, z = ((np.arange(n) + 0.5) * 2 * np.pi / n for n in (nx, ny, nz))
    C0 = 0.5 + 0.2 * np.cos(z)[:, None, None] * np.cos(2 * y)[None, :, None] * np.cos(x)[None, None, :]
    if bc[2] == D:
        C0 = (C0 - 0.5) * np.sin(z / 2)[:, None, None]
    C0 = C0.astype(np.float32).astype(np.float64)
    s = Solver(shape, h, bc, cn, pe, dt, C0, precision=prec)
    s.step(1)
    got = s.field()
    s.close()
    ref = co.step(C0, None, co.Params(nx, ny, nz, h, cn=cn, pe=pe, dt=dt, bc=bc), 1)
    # the bars of the other tests of the line solvers
    assert_parity(got, ref, 1e-12 if prec == "f64" else 1e-6, f"scans {shape} {bc} {prec}")
