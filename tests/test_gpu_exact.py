"""GPU tests of the FP64 / FP32 contraction through exact digit products.

The result is the rounded product of operands cut at 2^-63 (FP64) or 2^-39
(FP32) of their row's largest value, so beyond the modes' stated bars against
the oracle it has to be right where sums of digits reach their limits, at
every column-tile shape, and for the rows of C and AO values that the split
does not suit (those take fused multiply-adds).
"""
import ctypes
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


def _backward(m, W, C=None, points=None):
    from paper_2512_16677_gb300 import qmckl
    c = qmckl.Context("fp64")
    c.set_molecule(m)
    if C is not None:
        c.set_mo_coefficient(C)
    p = m.coord if points is None else points
    c.set_points_device(torch.from_numpy(np.ascontiguousarray(p)).cuda())
    dC, dR = c.backward_device(torch.from_numpy(np.ascontiguousarray(W)).cuda())
    torch.cuda.synchronize()
    c.synchronize()
    return dC.cpu().numpy(), dR.cpu().numpy()


@pytest.mark.parametrize("n_pts,n_mo", [(30, 6), (400, 17), (768, 33), (769, 100), (1601, 65)])
def test_backward_edges(orc, cfg, n_pts, n_mo):
    """FP64 backward around the edges of its slabs (768 points), k-steps and
    column parts, the weights of one component eight orders smaller (each
    component has exponents of its own), against the oracle's adjoint."""
    m = cfg(3, walk_num=9)
    rng = np.random.default_rng(n_pts)
    C = rng.normal(size=(n_mo, m.ao_num)) / np.sqrt(m.ao_num)
    mm = synth.Molecule(**{**m.__dict__, "mo_coef": C}).with_points(m.points[:n_pts])
    W = synth.random_weights(rng, n_pts, n_mo)
    W[:, 4] *= 1e-8
    dC, dR, sC, sR = orc.adjoint(mm, W, sizes=True)
    gC, gR = _backward(mm, W.reshape(1, n_pts, 5, n_mo))
    assert np.max(np.abs(gC - dC) / (sC + 1e-300)) <= 1e-12
    assert np.max(np.abs(gR - dR) / (sR + 1e-300)) <= 1e-12


def test_backward_weights_on_few_points_and_orbitals(orc, cfg):
    """Weights that are zero or tiny nearly everywhere take the multiply-adds
    and keep their accuracy relative to the terms that count."""
    m = cfg(3, walk_num=2)
    rng = np.random.default_rng(4)
    W = synth.random_weights(rng, m.point_num, m.mo_num)
    W[rng.random(m.point_num) < 0.9] *= 1e-11
    W[:, :, ::2] = 0.0
    dC, dR, sC, sR = orc.adjoint(m, W, sizes=True)
    gC, gR = _backward(m, W.reshape(m.walk_num, m.elec_num, 5, m.mo_num))
    assert np.max(np.abs(gC - dC) / (sC + 1e-300)) <= 1e-12
    assert np.max(np.abs(gR - dR) / (sR + 1e-300)) <= 1e-12


@pytest.mark.parametrize("config,walkers", [(2, 12), (5, 2)])
def test_backward_ranges_add_up(cfg, config, walkers):
    """Enough digits for several launch ranges of slabs (and of rows of W on
    the cluster): the gradient over all walkers is the sum of the halves'."""
    m = cfg(config, walk_num=walkers)
    h = walkers // 2
    g = torch.Generator(device="cuda").manual_seed(1)
    W = torch.rand((walkers, m.elec_num, 5, m.mo_num), dtype=torch.float64, device="cuda",
                   generator=g).sub_(0.5).cpu().numpy()
    whole = _backward(m, W)
    parts = [_backward(m, W[s], points=m.coord[s]) for s in (slice(0, h), slice(h, None))]
    for k in range(2):
        total = parts[0][k] + parts[1][k]
        scale = np.abs(parts[0][k]).max() + np.abs(parts[1][k]).max()
        assert np.abs(whole[k] - total).max() <= 1e-12 * scale


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("tiles,n_mo", [(303, 100), (304, 100), (320, 100), (610, 100), (620, 30)])
def test_many_items(cfg, mode, tiles, n_mo):
    """Around the count from which items are handed out as CTAs become free (608:
    304 tiles x 2 N tiles), an odd number of parts (3 in FP32: N tiles of unequal
    work that rotate), one N tile, and a ragged last tile.  Against the dense FP64
    AO values times C; bar: the mode's."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(2, walk_num=26)
    m = m.with_points(m.points[:25 * tiles - 3])
    C = np.random.default_rng(tiles).normal(size=(n_mo, m.ao_num)) / np.sqrt(m.ao_num)
    got = _mo(m, mode, C, points=m.coord)
    c = qmckl.Context("fp64")
    c.set_molecule(m)
    c.set_points_device(torch.from_numpy(m.coord).cuda())
    ao = c.ao_vgl_device().reshape(-1, m.ao_num)
    ct = torch.from_numpy(C.T.copy()).cuda()
    ref = (ao @ ct).cpu().numpy().reshape(got.shape)
    size = (ao.abs_() @ ct.abs_()).cpu().numpy().reshape(got.shape)
    c.synchronize()
    assert_within(mode, got, ref, size, f"{tiles} tiles, {n_mo} MOs")


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("config", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 26, 60, 280, 300, 620, 1300])
def test_small_calls_equal_large_ones(cfg, mode, config, n):
    """Calls of few blocks go without the reach pre-pass (up to 1300 blocks) and
    share a tile between the CTAs of a cluster (FP64 AO values: 4, 2 or 1 by the
    block count; digits: up to 8).  A point's outputs do not depend on that: the
    first n points alone equal the same points of a call of 20 000, bit for bit."""
    m = cfg(config, walk_num={1: 2000, 2: 34, 3: 100}[config])
    pts = m.points[:20000]
    big = _mo(m.with_points(pts), mode, points=pts)
    small = _mo(m.with_points(pts[:n]), mode, points=pts[:n])
    assert np.array_equal(big[:n], small)


@pytest.mark.parametrize("walkers", [1, 27])
def test_moves_through_tiles_equal_forward(cfg, walkers):
    """FP64 moves of a 500-AO basis (just past the line of the one-launch kernel) run
    through the tile kernels: equal, bit for bit, to a forward call at the proposed
    positions."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=walkers)
    pos = m.coord[:, 5] + 0.3
    c = qmckl.Context("fp64")
    c.set_molecule(m)
    c.set_points_device(torch.from_numpy(m.coord).cuda())
    c.set_single_point_device(5, torch.from_numpy(np.ascontiguousarray(pos)).cuda())
    got = c.mo_vgl_single_device()
    torch.cuda.synchronize()
    c.synchronize()
    assert np.array_equal(got.cpu().numpy(), _mo(m, "fp64", points=pos))


@pytest.mark.parametrize("mode,bits", [("fp64", 53), ("fp32", 24)])
@pytest.mark.parametrize("n", [16, 127, 144, 300, 1100])
def test_digit_sums_at_their_limits_of_either_sign(mode, bits, n):
    """The same operands with negative C, the first two thirds negative, and
    alternating signs: level sums far below zero, whose borrows run through
    every word of the integer sum."""
    v = sum(Fraction(127, 2 ** (8 * s + 7)) for s in range(1, 8)) + Fraction(63, 128)
    x = float(Fraction(int(v * 2 ** (bits + 1)), 2 ** (bits + 1)))
    sign = np.ones((3, n))
    sign[0] = -1.0
    sign[1, : 2 * n // 3] = -1.0
    sign[2, ::2] = -1.0
    got = _mo(_stack(x, n), mode, C=x * sign)[0, 0]
    for i in range(3):
        exact = int(sign[i].sum()) * Fraction(x) ** 2
        bar = n * Fraction(x) ** 2 / 2 ** bits * Fraction(17, 16)
        assert abs(Fraction(float(got[i])) - exact) <= bar, (i, float(got[i]), float(exact))


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("r", [0.0, 1.0])
def test_backward_digit_sums_at_their_limits(orc, sign, r):
    """Constant weights against constant coefficients and equal AOs, of equal and
    of opposite signs: long runs of equal products in dL/dC (points on the
    nucleus) and in W C (points a bohr away, seen through dL/dR)."""
    v = sum(Fraction(127, 2 ** (8 * s + 7)) for s in range(1, 8)) + Fraction(63, 128)
    x = float(Fraction(int(v * 2 ** 54), 2 ** 54))
    n, pts = 300, 320
    s = _stack(x, n)
    p = np.zeros((1, pts, 3))
    p[..., 0] = r
    m = synth.Molecule(**{**s.__dict__, "mo_coef": sign * x * np.ones((n, n))}).with_points(p[0])
    W = np.zeros((pts, 5, n))
    W[:] = x
    if r == 0.0:
        W *= sign
    dC, dR, sC, sR = orc.adjoint(m, W, sizes=True)
    gC, gR = _backward(m, W.reshape(1, pts, 5, n))
    assert np.max(np.abs(gC - dC) / (sC + 1e-300)) <= 1e-12
    assert np.max(np.abs(gR - dR) / (sR + 1e-300)) <= 1e-12


def _near_nuclei(m, rng, n, radii=(1e-3, 1e-2, 2e-2, 5e-2, 0.1)):
    """n points at each radius around randomly chosen nuclei, shuffled."""
    out = []
    for r in radii:
        v = rng.normal(size=(n, 3))
        v *= r / np.linalg.norm(v, axis=1, keepdims=True)
        out.append(m.nucl_coord[rng.integers(0, m.nucl_num, n)] + v)
    return rng.permutation(np.concatenate(out))


def _without(m, C, which, factor, rng):
    """C with the coefficients on every s shell, or on a fifth of the nuclei,
    multiplied by factor."""
    size = (m.shell_ang_mom + 1) * (m.shell_ang_mom + 2) // 2
    if which == "s shells":
        cols = np.repeat(m.shell_ang_mom == 0, size)
    else:
        some = rng.choice(m.nucl_num, max(1, m.nucl_num // 5), replace=False)
        cols = np.repeat(np.isin(m.shell_nucleus, some), size)
    C = np.array(C)
    C[:, cols] *= factor
    return C


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("config", [2, 3])
@pytest.mark.parametrize("which,factor", [("s shells", 0.0), ("nuclei", 0.0), ("nuclei", 1e-8),
                                          ("nuclei", 2e-3)])
def test_rows_dominated_by_an_absent_ao(orc, cfg, mode, config, which, factor):
    """MOs without the tight functions that dominate the AOs near a nucleus (nodes,
    pi orbitals): what is left is 8 orders below the row's exponent, and keeps
    the mode's accuracy.  A point's outputs do not depend on its tile."""
    rng = np.random.default_rng(config)
    m = cfg(config, walk_num=1)
    C = _without(m, rng.normal(size=(70, m.ao_num)) / np.sqrt(m.ao_num), which, factor, rng)
    pts = _near_nuclei(m, rng, 101)
    ref, size = orc.mo_vgl(m, points=pts, C=C)
    got = _mo(m, mode, C, pts[None])
    assert_within(mode, got, ref, size, f"{which} x {factor}")
    assert np.array_equal(_mo(m, mode, C, pts[None, ::3]), got[::3])


@pytest.mark.parametrize("config", [1, 3])
@pytest.mark.parametrize("factor", [0.0, 1e-8, 2e-3])
def test_backward_columns_dominated_by_a_weightless_point(orc, cfg, config, factor):
    """Points next to nuclei with zero or tiny weights: their AOs set the exponents of
    the columns of dL/dC, which consists of the other points' terms."""
    rng = np.random.default_rng(config)
    m = cfg(config, walk_num=40 if config == 1 else 4)
    near = _near_nuclei(m, rng, 35)
    pts = np.concatenate([m.points[:400], near])
    order = rng.permutation(len(pts))
    C = rng.normal(size=(33, m.ao_num)) / np.sqrt(m.ao_num)
    mm = synth.Molecule(**{**m.__dict__, "mo_coef": C}).with_points(pts[order])
    W = synth.random_weights(rng, len(pts), 33)
    W[400:] *= factor
    W = W[order]
    dC, dR, sC, sR = orc.adjoint(mm, W, sizes=True)
    gC, gR = _backward(mm, W.reshape(1, -1, 5, 33))
    assert np.max(np.abs(gC - dC) / (sC + 1e-300)) <= 1e-12
    assert np.max(np.abs(gR - dR) / (sR + 1e-300)) <= 1e-12


def test_backward_weights_on_the_smaller_orbitals(orc, cfg):
    """Weights on the half of the MOs whose coefficients are 12 orders below the other
    half's: W C, and with it dL/dR, consists of terms far below the exponents."""
    m = cfg(3, walk_num=2)
    rng = np.random.default_rng(8)
    C = rng.uniform(0.5, 1.0, size=(40, m.ao_num)) / np.sqrt(m.ao_num)
    C *= rng.choice([-1.0, 1.0], size=C.shape)
    C[1::2] *= 1e-12
    mm = synth.Molecule(**{**m.__dict__, "mo_coef": C})
    W = rng.uniform(0.5, 1.0, size=(m.point_num, 5, 40)) * rng.choice([-1.0, 1.0], size=(1, 5, 40))
    W[:, :, ::2] = 0.0
    dC, dR, sC, sR = orc.adjoint(mm, W, sizes=True)
    gC, gR = _backward(mm, W.reshape(m.walk_num, m.elec_num, 5, 40))
    assert np.max(np.abs(gC - dC) / (sC + 1e-300)) <= 1e-12
    assert np.max(np.abs(gR - dR) / (sR + 1e-300)) <= 1e-12


def test_refused_weights_cost_little(cfg):
    """Weights that do not suit the digits take the multiply-adds without the digit
    products before them: as long as with coefficients that are refused on the
    host (which launch no digit kernel), up to the pass over W that finds it out
    and some ten empty launches (2% of it)."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=8)
    rng = np.random.default_rng(5)
    W = synth.random_weights(rng, m.point_num, m.mo_num)
    W[rng.random(m.point_num) < 0.9] = 0.0
    dW = torch.from_numpy(W.reshape(m.walk_num, m.elec_num, 5, m.mo_num)).cuda()
    ctxs = []
    for C in (m.mo_coef, m.mo_coef * np.logspace(0, -8, m.mo_num)[:, None]):
        c = qmckl.Context("fp64")
        c.set_molecule(m)
        c.set_mo_coefficient(np.ascontiguousarray(C))
        c.set_points_device(torch.from_numpy(m.coord).cuda())
        c.mo_vgl_device()
        c.backward_device(dW)
        ctxs.append(c)
    times = ([], [])
    for _ in range(25):
        for c, t in zip(ctxs, times):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            c.backward_device(dW)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
    assert np.median(times[0]) <= 1.07 * np.median(times[1])


def test_digits_of_c_from_another_stream(cfg):
    """The digits that the first call after an upload of C makes on its stream are
    complete when it returns: a move on another stream, in a workspace of its
    own, may use them without waiting for the first."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=27)
    pos = torch.from_numpy(np.ascontiguousarray(m.coord[:, 3] + 0.2)).cuda()
    rng = np.random.default_rng(2)
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        C = rng.normal(size=m.mo_coef.shape) / np.sqrt(m.ao_num)
        c = qmckl.Context("fp64")
        c.set_molecule(m)
        c.set_mo_coefficient(C)
        c.set_points_device(torch.from_numpy(m.coord).cuda())
        c.set_single_point_device(3, pos)
        torch.cuda.synchronize()
        with torch.cuda.stream(one):
            c.mo_vgl_device()
        with torch.cuda.stream(two):
            got = c.mo_vgl_single_device()
        torch.cuda.synchronize()
        c.synchronize()
        want = c.mo_vgl_single_device()
        torch.cuda.synchronize()
        assert torch.equal(got, want)


def _captured(c, run):
    """run() captured into a graph after one call outside of it."""
    run()
    torch.cuda.synchronize()
    c.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        run()
    return g


def test_modes_keep_digits_of_their_own(cfg):
    """A call captured in FP64 reads the FP64 digits of C on every replay, whatever
    the context computed in FP32 since."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=2)
    c = qmckl.Context("fp64")
    c.set_molecule(m)
    p = torch.from_numpy(m.coord).cuda()
    c.set_points_device(p)
    out = torch.empty((2, m.elec_num, 5, m.mo_num), dtype=torch.float64, device="cuda")

    def run():
        c.set_points_device(p)
        c.mo_vgl_device(out=out)

    g = _captured(c, run)
    run()
    torch.cuda.synchronize()
    want = out.clone()
    c.set_compute_mode("fp32")
    c.mo_vgl_device()
    torch.cuda.synchronize()
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def _new_c(m, seed):
    return np.random.default_rng(seed).normal(size=m.mo_coef.shape) / np.sqrt(m.ao_num)


def test_replays_after_an_upload_read_its_digits(cfg):
    """Forward and backward calls captured in FP64 give the results of a newly uploaded
    C when they are replayed, also when the upload came with a call in FP32 or
    without a backward."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=2)
    p = torch.from_numpy(m.coord).cuda()
    W = torch.from_numpy(synth.random_weights(np.random.default_rng(1), m.point_num, m.mo_num)
                         .reshape(2, m.elec_num, 5, m.mo_num)).cuda()

    def new():
        c = qmckl.Context("fp64")
        c.set_molecule(m)
        c.set_points_device(p)
        return c

    c = new()
    out = torch.empty((2, m.elec_num, 5, m.mo_num), dtype=torch.float64, device="cuda")
    grads = []

    def forward():
        c.set_points_device(p)
        c.mo_vgl_device(out=out)

    def backward():
        grads[:] = c.backward_device(W)

    backward()  # (the largest workspace first: the graphs hold its address)
    gb = _captured(c, backward)
    captured = list(grads)
    gf = _captured(c, forward)
    for seed, mode in ((1, "fp64"), (2, "fp32")):
        C = _new_c(m, seed)
        c.set_mo_coefficient(C)
        c.set_compute_mode(mode)
        c.mo_vgl_device()
        c.set_compute_mode("fp64")
        gf.replay()
        gb.replay()
        torch.cuda.synchronize()
        r = new()
        r.set_mo_coefficient(C)
        want = r.mo_vgl_device()
        wC, wR = r.backward_device(W)
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        assert torch.equal(captured[0], wC) and torch.equal(captured[1], wR)


def test_capture_after_an_upload_takes_the_digits(cfg):
    """The digits come with the upload of C, whichever call brings it: a forward call
    captured after a density call rounds as an uncaptured one."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=2)
    p = torch.from_numpy(m.coord).cuda()
    c = qmckl.Context("fp64")
    c.set_molecule(m)
    c.set_points_device(p)
    out = torch.empty((2, m.elec_num, 5, m.mo_num), dtype=torch.float64, device="cuda")
    c.mo_vgl_device(out=out)
    C = _new_c(m, 3)
    c.set_mo_coefficient(C)
    c.density_device(np.ones(m.mo_num))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.set_points_device(p)
        c.mo_vgl_device(out=out)
    g.replay()
    torch.cuda.synchronize()
    got = out.clone()
    c.mo_vgl_device(out=out)
    torch.cuda.synchronize()
    assert torch.equal(got, out)


def _move_kernels(m, C, mode="fp64"):
    """Kernels of one single-electron move (after a first one) and its outputs."""
    from paper_2512_16677_gb300 import qmckl
    c = qmckl.Context(mode)
    c.set_molecule(m)
    c.set_mo_coefficient(np.ascontiguousarray(C))
    c.set_points_device(torch.from_numpy(m.coord).cuda())
    c.set_single_point_device(5, torch.from_numpy(np.ascontiguousarray(m.coord[:, 5] + 0.3)).cuda())
    c.mo_vgl_single_device()
    c.kernel_count()
    out = c.mo_vgl_single_device()
    n = c.kernel_count()
    torch.cuda.synchronize()
    c.synchronize()
    return n, out.cpu().numpy()


@pytest.mark.parametrize("config", [2, 3])
def test_moves_with_refused_c_take_one_launch(orc, cfg, config):
    """FP64 moves whose C does not suit the digits run in the one launch, which is
    several times faster than the tile kernels' multiply-adds (one AO and one
    contraction launch)."""
    m = cfg(config, walk_num=3)
    C = m.mo_coef * np.where(np.arange(m.ao_num) % 4 == 0, 1.0, 1e-6)
    n, got = _move_kernels(m, C)
    ref, size = orc.mo_vgl(m, points=m.coord[:, 5] + 0.3, C=C)
    assert_within("fp64", got, ref, size, "refused C")
    assert n == 1
    assert _move_kernels(m, m.mo_coef)[0] == 3


def test_products_on_two_streams(cfg):
    """A forward call and the moves of a large population, each with more items than
    a product hands out in fixed strides, at once on two streams (their workspaces
    are separate): each gives what it gives alone."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(2, walk_num=11)
    p = m.points[:6200].reshape(3100, 2, 3)
    c = qmckl.Context("fp64")
    c.set_molecule(m.with_points(p))
    c.set_points_device(torch.from_numpy(np.ascontiguousarray(p)).cuda())
    c.set_single_point_device(1, torch.from_numpy(np.ascontiguousarray(p[:, 1] + 0.2)).cuda())
    want = c.mo_vgl_device().clone(), c.mo_vgl_single_device().clone()
    torch.cuda.synchronize()
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(20):
        with torch.cuda.stream(one):
            a = c.mo_vgl_device()
        with torch.cuda.stream(two):
            b = c.mo_vgl_single_device()
        torch.cuda.synchronize()
        c.synchronize()
        assert torch.equal(a, want[0]) and torch.equal(b, want[1])


def test_captured_moves(cfg):
    """An FP64 move captured at a larger population than any move before, and a
    split-bf16 move whose graph is replayed after FP64 moves of the same context
    (the modes' workspaces are separate)."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=60)
    c = qmckl.Context("fp64")
    c.set_molecule(m)

    def propose(w):
        c.set_points_device(torch.from_numpy(np.ascontiguousarray(m.coord[:w])).cuda())
        c.set_single_point_device(2, torch.from_numpy(m.coord[:w, 2] + 0.2).cuda())

    propose(3)
    c.mo_vgl_single_device()
    propose(60)
    torch.cuda.synchronize()
    out = torch.empty((60, 5, m.mo_num), dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.mo_vgl_single_device(out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, c.mo_vgl_single_device())

    c.set_compute_mode("bf16x3")
    out32 = torch.empty((60, 5, m.mo_num), dtype=torch.float32, device="cuda")
    g32 = _captured(c, lambda: c.mo_vgl_single_device(out=out32))
    want = c.mo_vgl_single_device()
    c.set_compute_mode("fp64")
    c.mo_vgl_single_device()
    torch.cuda.synchronize()
    out32.zero_()
    g32.replay()
    torch.cuda.synchronize()
    assert torch.equal(out32, want)


def _workspace_call(c, out, ws):
    """qk_get_mo_vgl_device with a caller's workspace of exactly ws.numel() bytes."""
    c._check(c.lib.qk_set_workspace(c.h, ctypes.c_void_p(ws.data_ptr()), ws.numel()), "workspace")
    c._check(c.lib.qk_get_mo_vgl_device(c.h, ctypes.c_void_p(out.data_ptr()), out.numel()), "mo")
    c.synchronize()


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_smaller_workspaces(orc, cfg, mode):
    """A workspace with room for fewer digits than asked for: for some tiles, for one
    (same results), for none (multiply-adds, down to the AO tensor alone)."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(3, walk_num=5)
    c = qmckl.Context(mode)
    c.set_molecule(m)
    c.set_points_device(torch.from_numpy(m.coord).cuda())
    full = c.workspace_size()
    chunks = ctypes.c_int64()
    c._check(c.lib.qk_get_ao_chunk_num(c.h, ctypes.byref(chunks)), "chunks")
    tiles, nq, es = (m.point_num + 24) // 25, chunks.value, 8 if mode == "fp64" else 4

    def up(x):
        return (x + 255) // 256 * 256

    least = up(tiles * 128 * nq * 64 * es) + up(tiles * ((nq + 15) // 16 * 16)) + up(tiles * nq * 4)
    tile = 4 * nq * (32768 if mode == "fp64" else 20480)  # digits of a tile
    assert least + tiles * tile < full
    want = torch.empty((5, m.elec_num, 5, m.mo_num), dtype=c.dtype_torch, device="cuda")
    got = torch.empty_like(want)
    _workspace_call(c, want, torch.empty(full, dtype=torch.uint8, device="cuda"))
    ref, size = orc.mo_vgl(m)
    for extra in (7 * tile + 16384, 1 * tile + 16384, tile // 2, 0):
        got.zero_()
        ws = torch.empty(least + extra, dtype=torch.uint8, device="cuda")
        _workspace_call(c, got, ws)
        if extra >= tile:
            assert torch.equal(got, want)
        assert_within(mode, got.double().cpu().numpy().reshape(ref.shape), ref, size, f"+ {extra}")
    with pytest.raises(qmckl.QmcklError):
        _workspace_call(c, got, torch.empty(least - 256, dtype=torch.uint8, device="cuda"))
