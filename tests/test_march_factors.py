"""CPU tests of the marching line solver's constant factors and restart distance
(line_tables.h) and of the rule that picks a line solver (line_rule.h)."""
import numpy as np
import pytest

import _line_form as lf

CK = [1e-9, 0.02, 0.25, 1.2, 3.0, 12.0, 40.0, 400.0, 1e6]


@pytest.fixture(scope="module", autouse=True)
def _compiled():
    if lf.lib() is None:
        pytest.skip("no host C++ compiler")


@pytest.mark.parametrize("ck", CK)
def test_factors_multiply_to_the_operator(ck):
    l1, l2, dinv, _ = lf.factors("f64", ck)
    got = np.array([1 + l1 ** 2 + l2 ** 2, l1 * (1 + l2), l2]) / dinv
    # 1 / dinv = ck / l2 grows with ck, and the sums cancel against it
    assert np.abs(got - np.array([1 + 6 * ck, -4 * ck, ck])).max() <= 16 * 2.0 ** -53 * (1 + 16 * ck)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("ck", CK)
def test_restart_is_long_enough_and_no_longer(prec, ck):
    """What a start from zero `reach` rows early leaves of the recurrence is under 2^-64 (FP64) or 2^-36 (FP32),
    and 8 rows less would leave more; 0 where no distance up to the limit does."""
    l1, l2, _, reach = lf.factors(prec, ck)
    tol = 2.0 ** (-64 if prec == "f64" else -36)

    def left(rows):
        return np.abs(np.linalg.matrix_power(np.array([[-l1, -l2], [1.0, 0.0]]), rows)).max()

    rounding = 1 + 96 * 2.0 ** (-50 if prec == "f64" else -20)  # of l1 and l2, carried through the rows
    if reach:
        assert reach % 8 == 0 and left(reach) <= tol * rounding
        assert reach == 8 or left(reach - 8) * rounding > tol
    else:
        assert left(96) * rounding > tol


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_a_form_takes_only_lines_that_it_solves(prec):
    """Over random boxes: no form of a line shorter than its restart (none of a streamed block), no tile over its
    warps or its shared memory, and the scans wherever the operator decays too slowly."""
    rng = np.random.default_rng(2)
    block, esz = (64, 8) if prec == "f64" else (32, 4)
    taken = set()
    for _ in range(4000):
        shape = tuple(int(v) for v in np.exp(rng.uniform(np.log(5), np.log(1024), 3)))
        d, reach = int(rng.integers(3)), int(rng.integers(0, 13)) * 8
        f, us = lf.form(prec, rng.integers(2), d, shape, reach)
        n = shape[2 - d]
        taken.add(f)
        assert f in us and us[f] <= us["scan"]
        if reach == 0:
            assert f == "scan"
        if f == "march":
            assert n > -(-reach // block) * block
        if f.startswith("tile"):
            R = int(f[4:])
            warps = -(-(n + reach) // R)
            assert reach <= n and warps <= {16: 20, 32: 16, 64: 8}[R]
            assert (-(-warps * R // 32) * 32 + 16 // esz) * 32 * esz <= 227 * 1024
    assert taken == {"scan", "tile32", "march", "tile64" if prec == "f64" else "tile16"}


# solves where one form is far the fastest (us measured: scan, tile of 16 or 64 rows, tile of 32, streamed)
@pytest.mark.parametrize("prec, periodic, d, shape, reach, best", [
    ("f32", False, 2, (96, 512, 512), 72, "scan"),       # 95, 189, 157, 427
    ("f32", False, 1, (700, 80, 80), 72, "scan"),        # 28, 43, 35, 129
    ("f32", True, 0, (128, 256, 256), 16, "march"),      # 29, 27, 27, 16
    ("f32", True, 1, (512, 1024, 1024), 32, "march"),    # 1420, -, -, 648
    ("f64", True, 0, (1, 256, 256), 88, "scan"),         # 20, 41, 51, 117
    ("f64", False, 1, (1, 1024, 1024), 88, "scan"),      # 94, -, -, 407
    ("f64", True, 0, (700, 80, 80), 24, "tile64"),       # 463, 104, 106, 211
    ("f64", True, 0, (67, 131, 513), 24, "march"),       # 328, -, -, 183
])
def test_rule_on_clear_cases(prec, periodic, d, shape, reach, best):
    assert lf.form(prec, periodic, d, shape, reach)[0] == best


def test_oracle_boxes_take_every_form():
    """The boxes of test_gpu_march.py between them: forms x directions x copy widths x periodic lines and walls."""
    seen = set()
    for shape, prec, ck in lf.BOXES:
        nz, ny, nx = shape
        reach = lf.factors(prec, ck)[3]
        for d in range(3):
            aligned = (nx * ny if d == 2 else nx) * (4 if prec == "f32" else 8) % 16 == 0
            for per in (True, False):
                seen.add((prec, lf.form(prec, per, d, shape, reach)[0], d, aligned, per))
    want = {(prec, f, d, a, per) for prec, fs in (("f32", ("tile16", "tile32", "march")),
                                                  ("f64", ("tile32", "tile64", "march")))
            for f in fs for d in range(3) for a in (True, False) for per in (True, False)}
    want -= {("f32", "march", d, False, per) for d in (0, 2) for per in (True, False)}  # test_large_boxes_match_fp64
    assert not want - seen, sorted(want - seen)
