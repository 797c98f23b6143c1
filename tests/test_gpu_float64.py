"""The float64 path where its cheap forms meet their limits: densities far from 1, nodes
without a real sound speed, infinite values under the smoothness indicator."""
import numpy as np
import pytest

from paper_2004_08503_gb300 import inputs, sidp

pytestmark = pytest.mark.gpu


def waves(x, y, amp, seed=3):
    rng = np.random.default_rng(seed)
    a, b, c = rng.uniform(0, 6, 3)
    return inputs._cons(1.0 + amp * np.sin(6 * np.pi * x + a) * np.cos(4 * np.pi * y + b), 0.3 + amp * np.sin(4 * np.pi * y + c),
                        amp * np.cos(6 * np.pi * x + b), 1.0 + amp * np.cos(4 * np.pi * x + 6 * np.pi * y + a))


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0])
@pytest.mark.parametrize("size", [1e-17, 1e-13, 1e-9, 1e-5, 1.0, 1e5, 1e9, 1e13, 1e17])
def test_entropy_minimum_holds_at_every_density(size, gamma):
    """Density, momentum and energy scaled alike (the flow is the same), amplitudes from 1e-5 to 0.2, so that candidates
    lie just below the entropy bound by every amount: the float64 violation stays at its rounding, 1e-12."""
    for amp in (1e-5, 1e-3, 0.2):
        sv = sidp.Solver(law="euler", p=3, nx=12, ny=12, bc=("periodic",) * 4, gamma=gamma)
        x, y = sv.node_coords()
        sv.set_state(size * waves(x, y, amp))
        sv.step(12)
        d = sv.diag()
        sv.close()
        assert d["max_entropy_violation"] <= 1e-12, (amp, d["max_entropy_violation"])
        assert d["max_bound_violation"] <= 1e-12


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("limiter", ["none", "lo"])
@pytest.mark.parametrize("node", [0, 1, 4])
def test_negative_pressure_at_a_face_keeps_the_neighbours_speed(node, limiter, precision):
    """One node (a corner, a face node) with p < 0, as the unlimited scheme can produce: its sound speed is NaN,
    its faces take the neighbour's finite speed, and the time step and the stage stay finite, in both precisions."""
    sv = sidp.Solver(law="euler", p=3, nx=7, ny=6, domain=(0.0, 1.4, 0.0, 1.2), bc=("outflow",) * 4, limiter=limiter,
                     precision=precision)
    x, y = sv.node_coords()
    u = waves(x, y, 0.1)
    i = (2 * 7 + 3) * 16 + node
    u[3, i] = 0.3 * (u[1, i] ** 2 + u[2, i] ** 2) / u[0, i]
    v = np.ascontiguousarray(u, dtype=np.float64 if precision == "fp64" else np.float32)
    sidp.sidp_upload_state(sv.ctx, v.ctypes.data)  # set_state takes admissible states only
    dt = sv.compute_dt()
    assert 0.0 < dt < 1.0
    sv.stage(1, dt)
    got = sv.get_state(1)
    sv.close()
    assert np.all(np.isfinite(got))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("curved", [False, True])
def test_an_infinite_indicator_allows_no_flux(curved, precision):
    """An element with an infinite density has no indicator (infinity over infinity) and NaN bounds, which
    allow no antidiffusive flux: its nodes off the infinite one's lines take the low-order update, to 1e-12 of the
    state's size (float32: 2e-5)."""
    got = []
    for cfg in (dict(limiter="subcell", smoothness=dict(gmin=-0.5, gmax=2.5)), dict(limiter="lo")):
        sv = sidp.Solver(law="advection", p=3, nx=7, ny=6, domain=(0.0, 1.4, 0.0, 1.2), bc=("periodic",) * 4, beta=(0.7, -0.4),
                         precision=precision, **cfg)
        x, y = sv.node_coords()
        if curved:
            b = 0.02 * np.sin(2 * np.pi * x / 1.4) * np.sin(2 * np.pi * y / 1.2)
            sv.set_geometry(x + b, y + b)
        u = 1.0 + np.sin(9 * x) * np.cos(8 * y)
        base = (2 * 7 + 3) * 16
        u[base + 5] = np.inf
        v = np.ascontiguousarray(u[None], dtype=np.float64 if precision == "fp64" else np.float32)
        sidp.sidp_upload_state(sv.ctx, v.ctypes.data)
        sv.stage(1, 2e-3)
        got.append(sv.get_state(1)[0, base:base + 16].reshape(4, 4))
        sv.close()
    off = np.ix_([0, 2, 3], [0, 2, 3])
    a, b = got[0][off], got[1][off]
    assert np.all(np.isfinite(b)) and np.max(np.abs(a - b)) <= (1e-12 if precision == "fp64" else 2e-5) * 2.0
