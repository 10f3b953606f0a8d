"""GPU tests of the FP64 / FP32 contraction through exact digit products.

The result is the rounded product of operands cut at 2^-63 (FP64) or 2^-39
(FP32) of their row's largest value, so beyond the modes' stated bars against
the oracle it has to be right where sums of digits reach their limits, at
every column-tile shape, and for the rows of C and AO values that the split
does not suit (those take fused multiply-adds).
"""
from fractions import Fraction

import numpy as np
import pytest

from paper_2512_16677_gb300 import synth
from tolerances import assert_within

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2512_16677_gb300 import buildlib
    buildlib.build()


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


def _mo(m, mode, C=None, points=None, host=False):
    from paper_2512_16677_gb300 import qmckl
    c = qmckl.Context(mode)
    c.set_molecule(m)
    if C is not None:
        c.set_mo_coefficient(C)
    p = m.coord if points is None else points
    if host:
        c.set_points(p)
        return c.mo_vgl().astype(np.float64)
    c.set_points_device(torch.from_numpy(np.ascontiguousarray(p)).cuda())
    out = c.mo_vgl_device()
    torch.cuda.synchronize()
    c.synchronize()
    return out.double().cpu().numpy().reshape(-1, 5, out.shape[-1])


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("n_mo", [1, 16, 17, 33, 49, 64, 65, 97, 112, 113, 130])
def test_column_tiles(orc, cfg, mode, n_mo):
    """Column tiles of one and two parts, full and ragged, odd MO counts
    (stores of single values) and a ragged last point tile."""
    m = cfg(3, walk_num=1)
    pts = m.points[:133]
    C = np.random.default_rng(n_mo).normal(size=(n_mo, m.ao_num)) / np.sqrt(m.ao_num)
    ref, size = orc.mo_vgl(m, points=pts, C=C)
    assert_within(mode, _mo(m, mode, C, pts[None]), ref, size, f"{n_mo} MOs")


def _stack(value, n):
    """n equal s functions on one nucleus, each of the given value there, and
    one point on the nucleus: the MO value is n * value * C."""
    def one():
        return np.ones(n)

    return synth.Molecule(
        "stack", np.array([1.0]), np.zeros((1, 3)), np.zeros(n, dtype=np.int64),
        np.zeros(n, dtype=np.int32), np.ones(n, dtype=np.int64), one(), 0.5 * one(),
        value * one(), one(), one(), value * np.ones((3, n)), np.zeros((1, 1, 3)))


@pytest.mark.parametrize("mode,bits", [("fp64", 53), ("fp32", 24)])
@pytest.mark.parametrize("n", [16, 127, 129, 300, 1100])
def test_digit_sums_at_their_limits(mode, bits, n):
    """Operands whose digits are 63, 127, 127, ...: level sums beyond 2^22.
    The result is the exact product up to one rounding and the levels that
    are not formed (below 2^-36 and 2^-58 of it for these digits)."""
    v = sum(Fraction(127, 2 ** (8 * s + 7)) for s in range(1, 8)) + Fraction(63, 128)
    x = float(Fraction(int(v * 2 ** (bits + 1)), 2 ** (bits + 1)))
    exact = n * Fraction(x) ** 2
    got = _mo(_stack(x, n), mode)[0, 0]
    for g in got:
        assert abs(Fraction(float(g)) - exact) <= exact / 2 ** bits * Fraction(17, 16), float(g)


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_graded_coefficients(orc, cfg, mode):
    """MOs that live on a few AOs, with tails 12 orders smaller: a common
    exponent would lose the tails, whose own bar holds all the same."""
    m = cfg(3, walk_num=1)
    pts = m.points[::7]
    C = np.array(m.mo_coef)
    C[:, : m.ao_num // 2] *= 1e-12
    C[::2, :-20] *= 1e-12
    ref, size = orc.mo_vgl(m, points=pts, C=C)
    assert_within(mode, _mo(m, mode, C, pts[None]), ref, size, "graded C")


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_non_finite_values(orc, cfg, mode):
    """An infinite AO makes the rows it reaches what plain products make
    them; a coefficient beyond FP32 leaves the other MOs alone."""
    m = cfg(1)
    C = np.array(m.mo_coef)
    C[2, 5] = 1e300
    got = _mo(m, mode, C)
    ref, size = orc.mo_vgl(m, C=C)
    keep = [0, 1, 3, 4]
    assert_within(mode, got[:, :, keep], ref[:, :, keep], size[:, :, keep], "other MOs")
    n = 3
    s = _stack(1.0, n)
    s.shell_factor[1], s.coefficient[1] = 1e200, 1e200
    s.mo_coef[1] = -1.0
    with np.errstate(over="ignore"):
        v = _mo(s, mode, points=np.array([[[0.0, 0.0, 0.0], [1e3, 0.0, 0.0]]]))
    assert np.all(v[0, 0] == np.array([np.inf, -np.inf, np.inf]))
    assert np.all(v[1] == 0.0)


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_host_ranges_equal_device(cfg, mode):
    """The host call's point ranges and the one-launch path round the same
    exact sums: bit for bit equal."""
    m = cfg(3, walk_num=100)
    np.testing.assert_array_equal(_mo(m, mode, host=True), _mo(m, mode))
