"""The step kernels at the sizes and depths where their variants can go wrong,
against the FP64 oracle: films around the depth from which Eq. 14's velocity
factor is 1/h, tile edges and remainders, and non-finite states; the line
solves' FP64 digits and the single-precision results' bits.

Bars of the comparisons with the oracle: those of the parity tests, relative L2
1e-10 (FP64) and 1e-4 (FP32) for eta, ten times that for P and Q.
"""
import zlib

import numpy as np
import pytest

from paper_1611_05984_gb300 import scenarios as sc
from tests.helpers import oracle_from, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-10, "f32": 1e-4}


def _match(s, prec, steps):
    from paper_1611_05984_gb300 import celeris
    o = oracle_from(s)
    g = celeris.from_scenario(s, dtype=torch.float64 if prec == "f64" else torch.float32)
    o.step(steps)
    g.step(steps)
    ref = o.state()
    got = [a.double().cpu().numpy() for a in g.state()]
    assert rel_l2(got[0] - s.ws, ref[0] - s.ws) <= TOL[prec]
    for a, b in zip(got[1:], ref[1:]):
        if np.linalg.norm(b) > 1e-12:
            assert rel_l2(a, b) <= 10 * TOL[prec]


@pytest.mark.parametrize("friction", [0, 1, 2])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_films_around_the_desingularisation_depth(prec, friction):
    """Depths from 0 to three times eps^(1/4) over a bumpy bed, some cells dry
    and some a film: faces with both, one or no side past the threshold."""
    rng = np.random.default_rng(3)
    nx, ny, eps = 70, 45, 1e-4            # threshold depth 0.1 m
    s = sc.flat_basin(nx, ny, 1.0, 1.0, 0.004, model=1, K=0, friction=friction, fcoef=0.01, eps=eps)
    s.z = -0.3 + 0.25 * sc.random_bed(nx, ny, 5, 0.0, 1.0, smooth=2)
    s.w0 = s.z + np.maximum(rng.uniform(-0.05, 0.3, (ny, nx)), 0.0)
    s.P0 = 0.02 * rng.standard_normal((ny, nx))
    s.Q0 = 0.02 * rng.standard_normal((ny, nx))
    _match(s, prec, 3)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("field,value", [("w", np.inf)] + [(f, v) for f in "PQ" for v in (np.nan, -np.nan, np.inf)])
def test_a_non_finite_cell_reaches_its_neighbours(field, value, prec):
    """In shallow water nothing but the fluxes couples cells, so a non-finite
    value that leaves its neighbours finite was swallowed by a face.  After one
    step w is non-finite in the cell and in the neighbours whose mass flux the
    value enters (w: all four, P: west and east, Q: south and north), and
    finite three cells away.  (A NaN in w is raised to the bed when the state
    is set.)"""
    from paper_1611_05984_gb300 import celeris
    s = sc.flat_basin(96, 80, 1.0, 2.0, 0.01, model=1)
    s.P0 = np.full((80, 96), 0.1)
    s.Q0 = np.full((80, 96), -0.05)
    g = celeris.from_scenario(s, dtype=torch.float64 if prec == "f64" else torch.float32)
    state = dict(zip("wPQ", g.state()))
    state[field][40, 30] = value
    g.set_state(state["w"], state["P"], state["Q"])
    g.step(1)
    assert not g.check_finite()
    w = g.state()[0].cpu().numpy()
    hit = [(40, 30)] + [(40, 29), (40, 31)] * (field != "Q") + [(39, 30), (41, 30)] * (field != "P")
    assert not any(np.isfinite(w[c]) for c in hit), [w[c] for c in hit]
    w[38:43, 28:33] = 0.0
    assert np.isfinite(w).all()


# The FP32 stencil's tiles are 64 columns by 16 or 8 rows (by the number of
# tiles), the FP64 stencil's 32 columns by 32, 4 or 2 rows: one column or row
# short of, at and past their edges, odd widths (a lane's second cell outside),
# and each height.
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(2, 2), (63, 7), (64, 8), (65, 9), (66, 33), (127, 31), (129, 32), (191, 65),
                                   (705, 450), (1345, 1500)])
def test_tile_edges_and_remainders(prec, nx, ny):
    """Waves towards a beach, with a maker on the west, sponges and a dry
    shore, over the Euler start-up and full steps."""
    if prec == "f64" and nx * ny > 500000:
        nx, ny = 1025, 540                      # the FP64 stencil's 32-row tiles
    dx = max(1.0, 430.0 / nx)
    s = sc.beach(nx=nx, ny=ny, dx=dx, sponge=max(1, min(50, ny // 8)))
    x = (np.arange(nx) + 0.5) * dx
    y = (np.arange(ny) + 0.5) * dx
    s.w0 = np.maximum(s.z, 0.2 * np.sin(0.09 * x)[None, :] * np.cos(0.05 * y)[:, None])
    s.P0 = 0.5 * np.where(s.z < -0.5, s.w0, 0.0)
    s.Q0 = 0.2 * np.where(s.z < -0.5, s.w0, 0.0)
    _match(s, prec, 5)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,K", [(95, 71, 0), (33, 9, 1), (129, 65, 2)])
def test_checkpoints_of_identical_runs_are_identical(nx, ny, K, prec):
    """Odd widths: a checkpoint holds whole padded rows, and its padding is 0
    whatever the kernels left there (a lane's second cell beyond an odd width)
    and whatever the buffers held before."""
    from paper_1611_05984_gb300 import celeris

    def run(scale):
        s = sc.flat_basin(nx, ny, 1.0, 2.0, 0.01, K=K, friction=1, fcoef=0.01, eps=1e-8)
        s.w0 = scale * np.add.outer(np.sin(0.3 * np.arange(ny)), np.cos(0.2 * np.arange(nx)))
        s.P0 = s.Q0 = 0.3 * s.w0
        g = celeris.from_scenario(s, dtype=torch.float64 if prec == "f64" else torch.float32)
        g.step(5)
        return g.checkpoint().cpu().numpy()
    first = run(0.1)
    run(0.17)
    np.testing.assert_array_equal(run(0.1), first)
    es, px = (8, (nx + 31) // 32 * 32) if prec == "f64" else (4, (nx + 31) // 32 * 32)
    rows = first[256:256 + ny * px * es].view(np.float64 if prec == "f64" else np.float32).reshape(ny, px)   # w
    assert not rows[:, nx:].any()


@pytest.mark.parametrize("K,model", [(0, 0), (2, 0), (1, 1)])
def test_carries_correctors_and_shallow_water_across_tiles(K, model):
    """The predictor-only carries, two corrector stages and the shallow-water
    model on a grid of several FP32 tiles with makers on all sides."""
    s = sc.flat_basin(150, 70, 1.0, 1.0, 0.02, model=model, K=K, friction=1, fcoef=0.01, eps=1e-8)
    s.z = -1.0 + 0.3 * sc.random_bed(150, 70, 6, -1.0, 1.0, smooth=4)
    for side in (sc.W, sc.E, sc.S, sc.N):
        s.sides[side] = sc.Side(sc.SINE, 0, ((0.02, 3.0, 0.3 + side, 0.1 * side),))
    for prec in ("f32", "f64"):
        _match(s, prec, 6)


@pytest.mark.parametrize("nx,ny,dx,d", [(256, 32, 0.05, 1.0), (512, 64, 0.1, 1.0), (200, 40, 0.03, 0.32)])
def test_line_solves_keep_fp64_digits(nx, ny, dx, d):
    """One Euler step of a hump at rest: P is the x-solves' increment itself,
    against the same systems solved in extended precision.  A system of
    r = (B + 1/3) d^2 / dx^2 is ill-conditioned by 1 + 4 r for smooth solutions;
    the elimination in the kernel's order leaves 0.05 eps (1 + 4 r) or less, one
    on rows scaled by their pivots with coefficients folded per line twice as
    much (0.10, 0.10 and 0.05): the bar lies between."""
    from paper_1611_05984_gb300 import celeris
    wide = np.longdouble
    s = sc.flat_basin(nx, ny, dx, d, 0.2 * dx / np.sqrt(9.81 * d))
    s.w0 = np.broadcast_to(0.1 * np.exp(-(((np.arange(nx) + 0.5) / nx - 0.4) * 12.0) ** 2), (ny, nx)).copy()
    g = celeris.from_scenario(s, dtype=torch.float64)
    g.step(1)
    rhs = g.field("U").cpu().numpy().astype(wide)
    P = g.state()[1].cpu().numpy()
    r = (wide(s.Bd) + wide(1) / wide(3)) * wide(d) * wide(d) / (wide(dx) * wide(dx))
    b = np.full(nx, 1 + 2 * r)
    b[0] += r
    b[-1] += r
    c, x = np.zeros(nx, wide), np.zeros_like(rhs)
    for k in range(nx):
        a = -r if k else wide(0)
        pivot = b[k] - a * c[k - 1]
        c[k] = -r / pivot
        x[:, k] = (rhs[:, k] - a * x[:, k - 1]) / pivot
    for k in range(nx - 2, -1, -1):
        x[:, k] -= c[k] * x[:, k + 1]
    err = float(np.linalg.norm((P - x).astype(np.float64)) / np.linalg.norm(x.astype(np.float64)))
    bar = (0.035 if d < 1.0 else 0.075) * 2.0 ** -53 * float(1 + 4 * r)
    assert err <= bar, f"{err:.2e} above {bar:.2e}"


def pinned_scenario(nx, ny, K, model, friction):
    """A state made of integers over powers of two (the same bits on every
    machine): a bed that rises through the water, films up to the
    desingularisation depth, waves, a maker on the west, sponges south and
    north."""
    def field(seed, amplitude, smooth):
        v = np.random.default_rng(seed).integers(-2 ** 16, 2 ** 16, (ny, nx)).astype(np.float64) / 2.0 ** 16
        for _ in range(smooth):
            p = np.pad(v, 1, mode="edge")
            v = 0.25 * (p[:-2, 1:-1] + p[2:, 1:-1] + p[1:-1, :-2] + p[1:-1, 2:])
        return amplitude * v
    s = sc.flat_basin(nx, ny, 0.5, 1.0, 2.0 ** -7, model=model, K=K, friction=friction, fcoef=2.0 ** -7, eps=2.0 ** -13)
    slope = (np.arange(nx) - 0.75 * nx)[None, :] / nx
    s.z = np.maximum(1.5 * slope, -0.75) + field(1, 0.25, 2)
    wave = field(2, 0.25, 3)
    s.w0 = np.maximum(s.z + np.maximum(field(3, 0.125, 0), 0.0) * (s.z > -0.125), wave * (s.z <= -0.125))
    s.P0 = np.where(s.z < -0.25, 0.5 * wave + field(4, 0.0625, 1), 0.0)
    s.Q0 = np.where(s.z < -0.25, field(5, 0.0625, 1), 0.0)
    s.sides[sc.W] = sc.Side(sc.SINE, 0, ((0.0625, 4.0, 0.25, 0.5),))
    for side in (sc.S, sc.N):
        s.sides[side] = sc.Side(sc.SPONGE, 5)
    return s


PINNED = [((70, 45, 0, 0, 0), (1265626185, 2747069968, 2655919531)),
          ((150, 70, 1, 0, 2), (3123990259, 260540825, 3538570324)),
          ((131, 97, 2, 1, 1), (3843166897, 426282889, 291765706)),
          ((705, 450, 1, 0, 1), (2790344708, 1654164686, 3218525507)),
          ((1345, 1500, 1, 0, 2), (1983882001, 1767290283, 3360973068))]


@pytest.mark.parametrize("case,crc", PINNED)
def test_single_precision_bits(case, crc):
    """Six steps in single precision give the same bits as ever: where a
    discharge is a small difference of large terms its digits depend on the
    order of the operations, so a reordered stage shows as another result
    (reordered fluxes, dispersive terms and line solves moved the cross-tank
    discharge around a 1178 x 1178 island by 4e-5 of its norm).  The pins are
    checksums of w, P and Q from the kernels that took one cell per thread."""
    from paper_1611_05984_gb300 import celeris
    g = celeris.from_scenario(pinned_scenario(*case), dtype=torch.float32)
    g.step(6)
    fields = [a.cpu().numpy() for a in g.state()]
    assert all(np.isfinite(a).all() for a in fields)
    assert [zlib.crc32((a + np.float32(0)).tobytes()) for a in fields] == list(crc)   # -0 as 0


def _spread(lo, hi, n=200000):
    """Positive doubles of every exponent from 2^lo to 2^hi, the ends among them."""
    rng = np.random.default_rng(11)
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))
    return np.concatenate([x, [2.0 ** lo, 2.0 ** hi], np.ldexp(1.0, np.arange(lo, hi, max(1, (hi - lo) // 500)))])


# largest errors in units of the result's last place: the last operation of the
# reciprocal and of the root rounds once, and their remainders are e^3 and e^4 with
# e < 2^-20; x^(-1/3) adds two roundings in e = 1 - x r^3, a third of each
@pytest.mark.parametrize("op,lo,hi,ulp", [("reciprocal", -1021, 1021, 0.51), ("sqrt", -1074, 1023, 0.51),
                                          ("rcbrt", -126, 127, 1.7)])
def test_fp64_elementary_functions(op, lo, hi, ulp):
    """The FP64 kernels' own functions over the exponents they serve, against
    extended precision."""
    from paper_1611_05984_gb300 import celeris
    x = _spread(lo, hi)
    wide = x.astype(np.longdouble)
    ref = {"reciprocal": lambda: 1 / wide, "sqrt": lambda: np.sqrt(wide), "rcbrt": lambda: 1 / np.cbrt(wide)}[op]()
    got = celeris.arithmetic_selfcheck(op, torch.from_numpy(x).cuda()).cpu().numpy()
    err = (np.abs(got.astype(np.longdouble) - ref) / np.spacing(ref.astype(np.float64))).astype(np.float64)
    assert err.max() <= ulp, (err.max(), x[err.argmax()])


@pytest.mark.parametrize("depth,eps", [(1e-39, 1e-160), (1e-20, 1e-90)])
def test_manning_friction_below_single_precision(depth, eps):
    """Films thinner than single precision holds, deeper than eps^(1/4): the
    friction's h^(-7/3) takes the double-precision root, and the state stays
    finite and follows the oracle."""
    from paper_1611_05984_gb300 import celeris
    s = sc.flat_basin(40, 36, 1.0, 1.0, 1e-3, model=1, friction=2, fcoef=0.01, eps=eps)
    s.z[:, 20:] = 0.0
    s.w0 = np.where(s.z < 0.0, 0.0, depth)
    s.w0[:, 24:] = 0.0
    o = oracle_from(s)
    g = celeris.from_scenario(s, dtype=torch.float64)
    o.step(2)
    g.step(2)
    assert g.check_finite()
    for a, b in zip(g.state(), o.state()):
        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=0, atol=1e-12)


def test_fp64_root_at_the_ends():
    from paper_1611_05984_gb300 import celeris
    x = np.array([0.0, -0.0, np.inf, np.nan, -1.0, -np.inf])
    got = celeris.arithmetic_selfcheck("sqrt", torch.from_numpy(x).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, [0.0, 0.0, np.inf, np.nan, np.nan, np.nan])


def test_fp64_half_keeps_what_is_not_finite():
    from paper_1611_05984_gb300 import celeris
    x = np.concatenate([_spread(-1021, 1023), [0.0, np.inf, np.nan, np.finfo(np.float64).max, 5e-324, 2.0 ** -1022]])
    x = np.concatenate([x, -x])
    got = celeris.arithmetic_selfcheck("half", torch.from_numpy(x).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, np.where(np.abs(x) < 2.0 ** -1021, x, 0.5 * x))
