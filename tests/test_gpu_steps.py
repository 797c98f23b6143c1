"""Whole steps of a tiny mesh in one cluster launch: that this path runs, and what is particular to it (several launches
per call, the clock of moving boundaries, prescribed ghosts, debug capture, threads)."""
import threading

import numpy as np
import pytest

from paper_2004_08503_gb300 import inputs, sidp

pytestmark = pytest.mark.gpu


def waves(x, y, seed):
    rng = np.random.default_rng(seed)
    a, b, c = rng.uniform(0, 6, 3)
    return inputs._cons(1.0 + 0.2 * np.sin(5 * x + a) * np.cos(4 * y + b), 0.3 + 0.2 * np.sin(4 * y + c), 0.2 * np.cos(5 * x + b),
                        1.0 + 0.2 * np.cos(4 * x + 3 * y + a))


def make(precision, bc=("periodic",) * 4, p=3, nx=8, ny=6, stream=None, seed=1):
    sv = sidp.Solver(stream=stream, law="euler", p=p, nx=nx, ny=ny, domain=(0.0, 1.0, 0.0, ny / nx), bc=bc, precision=precision)
    sv.set_state(waves(*sv.node_coords(), seed))
    return sv


@pytest.mark.parametrize("stats", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p,nx,ny", [(1, 16, 16), (2, 12, 8), (3, 8, 8), (4, 8, 4), (5, 8, 4), (6, 4, 4), (7, 4, 4)])
def test_sixteen_tiles_take_the_cluster_launch(p, nx, ny, precision, stats):
    """Two steps under a caller's stream capture: ordinary launches would open a capture of their own there, which is an
    error, so that the call succeeds only where the cluster holds the mesh.  Replayed, it is two steps."""
    import torch
    s = torch.cuda.Stream()
    a, b = make(precision, p=p, nx=nx, ny=ny, stream=s), make(precision, p=p, nx=nx, ny=ny)
    for v in (a, b):
        v.set_stats(stats)
        v.step(1)
    g = torch.cuda.CUDAGraph()
    a.synchronize()
    with torch.cuda.graph(g, stream=s):
        a.step(2)
    with torch.cuda.stream(s):
        g.replay()
    b.step(2)
    a.synchronize()
    np.testing.assert_array_equal(a.get_state(0), b.get_state(0))
    assert a.diag()["t"] == b.diag()["t"]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_more_steps_than_one_launch_takes(precision):
    """257 steps in one call (two launches, 256 + 1) against single-step calls, bit for bit; then 300 more."""
    a, b = make(precision, nx=4, ny=4), make(precision, nx=4, ny=4)
    for n in (257, 300):
        a.step(n)
        for _ in range(n):
            b.step(1)
        np.testing.assert_array_equal(a.get_state(0), b.get_state(0))
    da, db = a.diag(), b.diag()
    assert da["steps"] == db["steps"] == 557 and da["t"] == db["t"] and da["last_dt"] == db["last_dt"]
    assert da["max_bound_violation"] == db["max_bound_violation"] and da["max_entropy_violation"] == db["max_entropy_violation"]


def stagewise(sv, n):
    """n steps of stages with the time step of compute_dt, the clock set before each."""
    t = 0.0
    for _ in range(n):
        sv.set_time(t)
        dt = sv.compute_dt()
        for k in (1, 2, 3):
            sv.stage(k, dt)
        t += dt
    return t, dt


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("side", ["moving split", "prescribed ghosts"])
def test_boundaries_in_the_cluster_launch(side, precision):
    """A split side that moves across face nodes within a step (its ghosts are taken at t^n, t^n + dt and t^n + dt/2),
    and prescribed ghosts, against the same steps stage by stage on the same tile; 1e-12 of the state's size, the
    library's parity bar (float32: 2e-5), the ghosts being discontinuous."""
    bc = ("outflow", "outflow", "outflow", "split") if side == "moving split" else ("exact", "outflow", "wall", "wall")
    a, b = make(precision, bc), make(precision, bc)
    left = inputs._cons(np.array(1.3), np.array(0.2), np.array(0.0), np.array(1.4)).ravel()
    right = inputs._cons(np.array(0.9), np.array(-0.1), np.array(0.1), np.array(0.8)).ravel()
    for v in (a, b):
        if side == "moving split":
            v.set_split("N", 0.31, 20.0, left, right)
        else:
            v.set_ghost("W", np.repeat(left[:, None], 6 * 4, axis=1))
        v.step(0)
    b.set_tile(3)
    a.step(4)
    t, dt = stagewise(b, 4)
    eps = np.finfo(float if precision == "fp64" else np.float32).eps
    d = a.diag()
    assert abs(d["t"] - t) <= 8 * eps * t and abs(d["last_dt"] - dt) <= 64 * eps * dt
    ua, ub = a.get_state(0), b.get_state(0)
    assert np.max(np.abs(ua - ub)) <= (1e-12 if precision == "fp64" else 2e-5) * np.max(np.abs(ub))
    if side == "moving split":  # the boundary did move: frozen at its start the result is another one
        c = make(precision, bc)
        c.set_split("N", 0.31, 0.0, left, right)
        c.step(4)
        assert np.max(np.abs(ua - c.get_state(0))) > 1e-3


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_debug_capture_in_the_cluster_launch(precision):
    """Bounds, K and alpha of the last stage: those of the stage by itself."""
    a, b = make(precision), make(precision)
    for v in (a, b):
        v.set_debug(True)
    b.set_tile(3)
    a.step(2)
    stagewise(b, 2)
    tol = 1e-12 if precision == "fp64" else 2e-5
    for k, v in a.bounds().items():
        w = b.bounds()[k]
        err = np.abs(v - w) / np.max(np.abs(w))
        assert (np.mean(err <= tol) >= 0.98) if k == "alpha" else np.max(err) <= tol, (k, np.max(err))


def test_threads_each_with_its_own_mesh():
    """First launches of several clusters from threads of their own (each asks whether the device holds its cluster)."""
    sizes = [(2, 9, 6), (3, 6, 6), (3, 8, 4), (4, 6, 4), (5, 6, 4), (6, 4, 3), (2, 9, 8), (3, 8, 8)]
    got = [None] * len(sizes)

    def work(i):
        p, nx, ny = sizes[i]
        sv = make("fp64", p=p, nx=nx, ny=ny, seed=i)
        sv.step(5)
        got[i] = sv.get_state(0)
        sv.close()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, (p, nx, ny) in enumerate(sizes):
        sv = make("fp64", p=p, nx=nx, ny=ny, seed=i)
        sv.step(5)
        np.testing.assert_array_equal(got[i], sv.get_state(0))
        sv.close()
