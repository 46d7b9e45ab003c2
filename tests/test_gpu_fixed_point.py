"""The FP64 element kernels' fixed-point contractions against the oracle, at
the sizes and magnitudes where they could go wrong: every order with element
counts that leave the last CTA partly filled, equation groups of very
different magnitude, values beyond the fixed-point range (plain FP64 then),
and non-finite elements beside finite ones.

Bar: 1e-12 of the largest tendency of each variable, the FP64 bar of one
right-hand side (the integers hold 58 bits of each group's largest value, so
the contraction adds less than FP64's own rounding)."""
import numpy as np
import pytest

from paper_1511_01561_gb300 import inputs as I

from .helpers import lobatto_derivative, scaled_random_state
from .thin_box import thin_flow, thin_rhs

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def numa():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_01561_gb300 import build
    build.build()
    from paper_1511_01561_gb300 import numa as mod
    return mod


def _rhs(numa, cfg, q):
    s = numa.Solver(cfg, "fp64")
    try:
        return s.rhs(q).cpu().numpy()
    finally:
        s.close()


def _check(Rg, Ro):
    scale = np.abs(Ro).max(axis=1)
    scale[1:4] = scale[1:4].max()
    err = np.abs(Rg - Ro).max(axis=1) / np.where(scale > 0.0, scale, 1.0)
    assert err.max() <= TOL, err


# element counts that are no multiple of any number of elements per CTA, one
# element, thin slabs of unlike widths
@pytest.mark.parametrize("N", range(1, 9))
@pytest.mark.parametrize("ne,per", [((3, 1, 1), (0, 0, 0)), ((1, 1, 1), (0, 1, 0)), ((2, 3, 3), (1, 0, 0))])
def test_rect_orders_and_remainders(numa, orc, N, ne, per):
    cfg = I.box(ne, N, L=(3000.0, 700.0, 900.0), periodic=per)
    m = orc.Mesh(cfg)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=N)
    _check(_rhs(numa, cfg, q), m.rhs(q))


# the per-node form: warped boxes and the box's elements taken as curved, with
# rows of the metric 100 times apart
@pytest.mark.parametrize("N", range(1, 9))
@pytest.mark.parametrize("over", [dict(warp=0.04), dict(metric_form="nodal")], ids=["warped", "nodal"])
@pytest.mark.parametrize("ne,per", [((3, 1, 1), (0, 0, 0)), ((2, 3, 3), (1, 0, 0))])
def test_nodal_orders_and_remainders(numa, orc, N, ne, per, over):
    cfg = I.box(ne, N, L=(30000.0, 700.0, 900.0), periodic=per, **over)
    m = orc.Mesh(cfg)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=N)
    _check(_rhs(numa, cfg, q), m.rhs(q))


@pytest.mark.parametrize("N", [2, 4, 7])
@pytest.mark.parametrize("over", [dict(), dict(warp=0.03)], ids=["rect", "warped"])
@pytest.mark.parametrize("scale", [1e-30, 1e-200, 1e-310])
def test_small_momentum(numa, orc, N, over, scale):
    """The mass equation is linear in U: a momentum far below the other groups
    (1e-30), below the fixed-point range (1e-200) and subnormal (1e-310)."""
    cfg = I.box((3, 2, 2), N, **over)
    m = orc.Mesh(cfg)
    q = np.zeros((5, m.Ng))
    q[1:4] = np.random.default_rng(N).uniform(-1.0, 1.0, (3, m.Ng)) * scale
    Rg, Ro = _rhs(numa, cfg, q)[0], m.rhs(q)[0]
    tiny = 64 * 5e-324 if scale < 1e-300 else 0.0  # subnormal sums are rounded to whole units of 5e-324
    assert np.abs(Rg - Ro).max() <= TOL * np.abs(Ro).max() + tiny


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_rect_nonfinite_elements(numa, orc, bad):
    """One node's x momentum is not finite: the mass tendency is not finite on
    its x line inside its element and nowhere else (K_d D has no other term
    with U_x), and the nodes of the other elements are untouched."""
    cfg = I.box((4, 3, 3), 4)
    m = orc.Mesh(cfg)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=11)
    R0 = _rhs(numa, cfg, q)
    g = 5 + 17 * (6 + 13 * 6)
    q[1, g] = bad
    Rg = _rhs(numa, cfg, q)
    line = np.zeros(m.Ng, dtype=bool)
    line[g - 1:g + 4] = True  # ix = 4 .. 8
    assert np.array_equal(~np.isfinite(Rg[0]), line)
    e = m.l2g().reshape(-1, 125)
    near = np.unique(e[(e == g).any(axis=1)])
    far = np.setdiff1d(np.arange(m.Ng), near)
    assert np.array_equal(Rg[:, far], R0[:, far])


# columns of 61 and 64 levels (the tallest solved with the inverse) and of 65
# and 73 (the LU factors), at a vertical acoustic Courant number of 2 to 4
@pytest.mark.parametrize("N,nez", [(4, 15), (7, 9), (4, 16), (8, 9)])
def test_imex_column_heights(numa, orc, N, nez):
    from oracle import imex

    cfg = I.box((2, 1, nez), N, L=(4000.0, 2000.0, 250.0 * nez))
    ic = ("bubble", (0.5, 600.0, 2000.0, 1000.0, 120.0 * nez))
    dt = 3.0 * 250.0 * 0.5 * (1.0 - np.cos(np.pi / N)) / 350.0
    m = orc.Mesh(cfg)
    q = m.init_state(*ic)
    q[1:4] += np.random.default_rng(N).uniform(-0.1, 0.1, (3, m.Ng))
    qo, _ = imex.run_imex(m, q, dt, 3, 0.1)
    s = numa.Solver(cfg, "fp64")
    try:
        s.set_time_scheme("imex")
        s.set_robert_asselin(0.1)
        s.set_state(q)
        s.run(dt, 3)
        qg = s.get_state().numpy()
    finally:
        s.close()
    err = np.abs(qg - qo).max(axis=1) / np.maximum(np.abs(qo).max(axis=1), 1e-30)
    assert err.max() <= 1e-10, err


# the equation of state of the update's primitive pass: |Theta'/Theta0| within
# a factor 1.5 of 2^-k, both signs, zeros between them, on both sides of every
# term count and of the end of the integer form (2^-5).  At rest without a
# density perturbation the momentum tendency is the gradient of p' alone,
# which is proportional to Theta' for small ratios: its error relative to its
# own largest value is that of p'.
@pytest.mark.parametrize("prec", ["fp64", "fp64_pairs"])
@pytest.mark.parametrize("k", [1, 4, 5, 6, 10, 12, 15, 20, 30, 40, 60, 300, 900])
def test_pressure_over_magnitudes(numa, orc, prec, k):
    cfg = I.box((3, 2, 2), 4)
    m = orc.Mesh(cfg)
    rng = np.random.default_rng(k)
    q = np.zeros((5, m.Ng))
    x = np.ldexp(rng.uniform(0.5, 1.5, m.Ng), -k) * rng.choice([-1.0, 0.0, 1.0], m.Ng)
    q[4] = x * m.ref()[1]
    s = numa.Solver(cfg, prec)
    try:
        Rg = s.rhs(q).cpu().numpy()
    finally:
        s.close()
    _check(Rg, m.rhs(q))


# U, u and p' within 2^-31 below powers of two at every node: the diagonal
# momentum flux at its bound, where sums of two nodes' high halves are largest
@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("over", [dict(), dict(metric_form="nodal")], ids=["rect", "nodal"])
def test_momentum_flux_at_its_bound(numa, orc, N, axis, over):
    cfg = I.box((2, 2, 2), N, periodic=(1, 1, 0), **over)
    m = orc.Mesh(cfg)
    rho0, th0, p0 = m.ref()[:3]
    q = np.zeros((5, m.Ng))
    q[0] = 1.0 - rho0
    q[1 + axis] = 2.0 - 2.0 ** -40
    q[4] = th0 * np.expm1(np.log1p((4.0 - 2.0 ** -34) / p0) * cfg["cv"] / cfg["cp"])
    # uniform fluxes: the tendencies are zero but for the buoyancy, so each variable's
    # scale is its flux over an element's half edge
    scale = np.array([2.0, 8.0, 8.0, 8.0, 2.0 * 300.0]) / 250.0
    err = np.abs(_rhs(numa, cfg, q) - m.rhs(q)).max(axis=1) / scale
    assert err.max() <= TOL, err


# several elements share a CTA at N <= 3: one that the integers cannot hold
# (momentum of 1e200 at its nodes) leaves the bits of the others alone
@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("over", [dict(), dict(warp=0.03)], ids=["rect", "warped"])
def test_elements_of_one_cta_are_independent(numa, orc, N, over):
    cfg = I.box((11, 3, 3), N, **over)
    m = orc.Mesh(cfg)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=N)
    R0 = _rhs(numa, cfg, q)
    nx = 11 * N + 1
    g = 4 * N + 1 + nx * (N + (3 * N + 1) * N)  # on an edge between elements in y and z
    q[1, g] = 1e200
    Rg = _rhs(numa, cfg, q)
    e = m.l2g().reshape(-1, (N + 1) ** 3)
    far = np.setdiff1d(np.arange(m.Ng), np.unique(e[(e == g).any(axis=1)]))
    assert np.array_equal(Rg[:, far], R0[:, far])


# the same through slabs of an odd number of elements, which group the elements
# of a CTA otherwise: elements with a momentum below the integers' range ahead
# of a disturbance
@pytest.mark.parametrize("N,ne", [(1, (13, 11, 6)), (2, (7, 9, 6)), (3, (5, 5, 6))])
@pytest.mark.parametrize("over", [dict(), dict(warp=0.02)], ids=["rect", "warped"])
def test_slabs_with_elements_out_of_range(numa, orc, N, ne, over):
    cfg = I.box(ne, N, **over)
    m = orc.Mesh(cfg)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=N)
    ahead = m.coords()[2] > 420.0  # (of 1000)
    q[:, ahead] = 0.0
    q[1:4, ahead] = np.random.default_rng(N).uniform(-1e-200, 1e-200, (3, int(ahead.sum())))
    out = []
    for slabs in (1, 2, 3):
        s = numa.Solver(cfg, "fp64")
        try:
            assert s.set_slabs(slabs) == slabs
            s.set_state(q)
            s.run(1e-3, 1)
            out.append(s.get_state().numpy().copy())
        finally:
            s.close()
    assert np.array_equal(out[1], out[0]) and np.array_equal(out[2], out[0])


# densities within 2^-20 of 1, 1/2 and 1/4, on both sides: 1/rho next to the ends
# of its binade
@pytest.mark.parametrize("over", [dict(), dict(warp=0.03)], ids=["rect", "warped"])
def test_densities_next_to_powers_of_two(numa, orc, over):
    cfg = I.box((4, 3, 3), 4, **over)
    m = orc.Mesh(cfg)
    rng = np.random.default_rng(20)
    q = scaled_random_state(m.Ng, m.ref()[0], m.ref()[1], seed=20)
    d = np.ldexp(rng.uniform(0.5, 1.0, m.Ng), -rng.integers(20, 53, m.Ng)) * rng.choice([-0.5, 0.0, 1.0], m.Ng)
    q[0] = (1.0 + d) * rng.choice([1.0, 0.5, 0.25], m.Ng) - m.ref()[0]
    _check(_rhs(numa, cfg, q), m.rhs(q))


# a state at rest on meshes whose tables' power of two runs over the range in
# which a factor of a group of zeros came out as an infinity
@pytest.mark.parametrize("s2", range(98, 116))
def test_rest_on_tiny_elements(numa, orc, s2):
    N = 4
    row = max(float(sum(abs(v) for v in r)) for r in lobatto_derivative(N))
    h = np.sqrt(4.0 * 0.75 * 2.0 ** (60 - s2) / row)  # the largest row sum of h^2 / 4 |D|: 0.75 2^(60 - s2)
    cfg = I.box((3, 2, 2), N, L=(3 * h, 2 * h, 2 * h))
    R = _rhs(numa, cfg, np.zeros((5, orc.Mesh(cfg).Ng)))
    assert np.array_equal(R, np.zeros_like(R))


# 1D-IMEX through run and rk_step in any division into calls, with a new time
# step in between and a run of no steps first: the same states bit for bit (the
# columns' inverses are made when a step first needs them)
@pytest.mark.parametrize("nez", [3, 12, 17])
def test_imex_calls_in_any_division(numa, nez):
    cfg = I.box((2, 2, nez), 4, L=(4000.0, 4000.0, 250.0 * nez))

    def go(*calls):
        s = numa.Solver(cfg, "fp64")
        try:
            s.set_time_scheme("imex")
            s.init_state("bubble", (0.5, 600.0, 2000.0, 2000.0, 120.0 * nez))
            for dt, n, graph in calls:
                if graph:
                    s.run(dt, n)
                else:
                    for _ in range(n):
                        s.rk_step(dt)
            return s.get_state().numpy().copy()
        finally:
            s.close()

    a = go((0.2, 3, True), (0.1, 2, True), (0.2, 1, True))
    assert np.isfinite(a).all() and np.abs(a).max() > 0.0
    assert np.array_equal(a, go((0.2, 3, False), (0.1, 2, False), (0.2, 1, False)))
    assert np.array_equal(a, go((0.2, 0, True), (0.2, 1, True), (0.2, 2, True), (0.1, 1, False), (0.1, 1, True), (0.2, 1, True)))


# elements much wider than high (or higher than wide), each variable against its
# own rounding scale u S (thin_box.thin_rhs): FP64 arithmetic in the oracle's
# order stays within 1.2 u S on these states; the bar is twice u S
@pytest.mark.parametrize("over", [dict(), dict(metric_form="nodal")], ids=["rect", "nodal"])
@pytest.mark.parametrize("N", [2, 4, 5, 8])
@pytest.mark.parametrize("aspect", [0.01, 1.0, 16.0, 100.0, 500.0, 2500.0])
def test_thin_elements(numa, orc, aspect, N, over):
    h = 1e4 if aspect > 1.0 else 100.0 if aspect < 1.0 else 1e3
    cfg = I.box((3, 2, 2), N, L=(3.0 * h, 2.0 * h, 2.0 * h / aspect), **over)
    m = orc.Mesh(cfg)
    q = thin_flow(m, cfg)
    R, S = thin_rhs(m, cfg, q)
    err = np.abs(_rhs(numa, cfg, q) - R).max(axis=1).astype(float) / (2.0 ** -53 * S)
    assert err.max() <= 2.0, err
