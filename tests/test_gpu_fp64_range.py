"""The FP64 form far from one and on non-physical values.

States related by a similarity (rho, p and B^2 by powers of ten, u^2 by p / rho)
advance alike at any scale at which the squared speeds are representable, against
the CPU oracle.  Tolerance as for states near one: about 50 dependent operations
per cell and stage, 4 stages, each rounded once (2^-53): 50 x 4 x 1.1e-16 = 2.2e-14
if all errors add up: 1e-13 of a variable's largest value.

A NaN speed of one side of a face (a negative density): Rusanov takes the right
side's if the left one's is NaN and NaN if the right one's is, as the oracle does;
HLL and Linde take the other side's, or none where there is no other.  So the same
calls are non-physical as before the speeds were reformulated.

The operations themselves: 1/x outside the normal range is the division's value;
the fast speed is the usual form's, to 6.3 u where its inner root is not small
(u = 2^-53; both forms: the sums' 2 u, 9 u of the inner root's argument halved by
the roots: at most 6.2 u), NaN where that is NaN."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FLUXES = [W.FLUX_RUSANOV, W.FLUX_HLL, W.FLUX_LINDE]
SCALES = [(1e-100, 1e-100), (1e-160, 1e-160), (1e-290, 1e-290), (1e160, 1e160), (1e290, 1e290), (1.0, 1e-140),
          (1.0, 1e140), (1e-150, 1e-170), (1e290, 1e200)]


def _grid(rho_scale=1.0, p_scale=1.0, bc=W.BC_PERIODIC, flux=0, **more):
    root = (2, 2, 2)
    q = W.Problem("range", (-1.0,) * 3, (1.0,) * 3, root, W.as_leaf_array(W.uniform_leaves(root)), (bc,) * 6, flux=flux,
                  **more)
    x = W.cell_centres(q.lo, q.hi, root, q.leaves)
    s = [np.sin(np.pi * (a + 0.1 * k)) for k, a in enumerate(x)]
    u, b = np.sqrt(p_scale / rho_scale), np.sqrt(p_scale)
    return W.with_state(q, [rho_scale * (1 + 0.3 * s[0] * s[1]), u * 0.5 * s[1], u * 0.4 * s[2], u * 0.3 * s[0],
                            b * 0.5 * s[2], b * 0.4 * s[0], b * (0.6 + 0.2 * s[1]), p_scale * (1 + 0.3 * s[2])])


def _scaled_error(U, Uo):
    scale = np.abs(Uo).reshape(8, -1).max(1)
    for c in ((1, 2, 3), (4, 5, 6)):  # a component near zero against its vector's largest
        scale[list(c)] = scale[list(c)].max()
    return (np.abs(U - Uo).reshape(8, -1).max(1) / scale).max()


def _step(q, dt=None):
    """(status code, state, dt of the start) after two CFL steps or one of dt."""
    with bats.Solver(q) as h:
        h.set_state(0, q.U0)
        dt0, code = h.dt(0, 0.3), 0
        try:
            h.step_dt(1, dt) if dt else h.step(2, 0.3)
        except bats.BatsError as e:
            code = e.code
        return code, h.get_state(0), dt0


@pytest.mark.parametrize("flux", FLUXES)
@pytest.mark.parametrize("scale", SCALES)
def test_similar_states_advance_alike(scale, flux):
    q = _grid(*scale, flux=flux)
    Uo, dto, _ = O.run(q, q.U0, 2, cfl=0.3)
    assert np.all(np.isfinite(Uo))
    code, U, dt0 = _step(q)
    assert code == 0
    assert abs(dt0 / (0.3 / O.cfl_smax(q, q.U0)) - 1) <= 1e-14
    assert _scaled_error(U, Uo) <= 1e-13


@pytest.mark.parametrize("flux", FLUXES)
@pytest.mark.parametrize("side", range(6))
def test_inflow_of_negative_density(side, flux):
    q = _grid(flux=flux)
    bc = [W.BC_OUTFLOW] * 6
    bc[side] = W.BC_INFLOW
    q.bc = tuple(bc)
    q.inflow = np.array([-0.5, 0.1, 0.2, 0.1, 0.1, 0.2, 0.1, 1.0])
    code, U, _ = _step(q, 1e-3)
    if flux != W.FLUX_RUSANOV:
        assert code == 0 and np.all(np.isfinite(U))
        return
    Uo, _, _ = O.run(q, q.U0, 1, dt=1e-3)
    if np.all(np.isfinite(Uo)):
        assert code == 0 and _scaled_error(U, Uo) <= 1e-13
    else:
        assert code == bats.BATS_ERR_NONPHYSICAL
        assert np.array_equal(np.isfinite(U), np.isfinite(Uo))


@pytest.mark.parametrize("var,value,flux", [(0, -0.5, 0), (0, -0.5, 1), (0, -0.5, 2), (0, 0.0, 0), (0, 0.0, 1), (0, 0.0, 2),
                                            (0, np.nan, 0), (0, np.nan, 1), (0, np.nan, 2), (1, np.inf, 0), (1, np.inf, 1),
                                            (7, -1.0, 0), (7, -1.0, 1), (7, -1.0, 2), (7, np.nan, 0), (7, np.nan, 1)])
def test_a_non_physical_cell(var, value, flux):
    q = _grid(flux=flux)
    U0 = q.U0.copy()
    U0[var, 3, 3, 4, 5] = value
    q.U0 = U0
    code, U, _ = _step(q, 1e-5)
    assert code == bats.BATS_ERR_NONPHYSICAL
    Uo, _, _ = O.run(q, U0, 1, dt=1e-5)
    assert np.array_equal(np.isfinite(U), np.isfinite(Uo))


def test_operations_far_from_one():
    tiny = np.finfo(float).tiny
    x = np.array([0.0, -0.0, 5e-324, -5e-324, 1e-310, tiny, np.nextafter(tiny, 0), 2.0 ** 1021, 2.0 ** 1022, 1.7e308, -1.7e308,
                  np.inf, -np.inf, np.nan])
    with np.errstate(all="ignore"):
        rcp = bats.bats_debug_fp64_ops(np.ones_like(x), x)
        assert np.array_equal(rcp[0], 1 / x, equal_nan=True)
        assert np.array_equal(rcp[3], 1 / x, equal_nan=True)  # the velocity 1 / x
    assert bats.bats_debug_fp64_ops([0.0], [0.0])[1][0] == 0.0
    assert np.isnan(bats.bats_debug_fp64_ops([0.0], [-1.0])[1][0])

    rng = np.random.default_rng(7)
    n = 200000
    v = lambda lo, hi: np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))
    rho = v(-960, 960)
    e = np.clip(np.frexp(rho)[1] + rng.integers(-480, 480, n), -960, 960)
    g = np.ldexp(rng.uniform(1.0, 2.0, n), e)
    b = g * v(-6, 6)
    L = np.longdouble
    G = g.astype(L) + b.astype(L) / 2
    c = (rng.uniform(0, 1, n) * np.minimum(b.astype(L), 0.74 * G * G / (2 * g.astype(L)))).astype(float)
    got = bats.bats_debug_fp64_ops(g, rho, b, c)[4]
    exact = np.sqrt((G + np.sqrt(G * G - 2 * g.astype(L) * c.astype(L))) / rho.astype(L))
    assert float(np.max(np.abs(got.astype(L) / exact - 1))) <= 6.3 * 2.0 ** -53

    # signs and NaN as in the usual form
    vals = np.array([-1.0, 0.0, 0.3, 2.0, np.nan, np.inf])
    g, rho, bn, bt = (t.reshape(-1) for t in np.meshgrid(vals, vals, vals, vals))
    b, c = bn * bn + bt * bt, bn * bn
    with np.errstate(all="ignore"):
        a2 = 2 * g / rho
        s = a2 + b / rho
        disc = s * s - 4 * a2 * (c / rho)
        want = np.sqrt(0.5 * (s + np.sqrt(np.where(disc < 0, 0.0, disc))))
    got = bats.bats_debug_fp64_ops(g, rho, b, c)[4]
    assert np.array_equal(np.isnan(got), np.isnan(want))
