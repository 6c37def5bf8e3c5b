"""Whole-instance solves of 1D problems (one launch per solve, the iterates in
shared memory) against the same handle iterating with one launch per
iteration (use_graph=0): the same arithmetic in the same order, so the same
iteration counts and status, and solutions that agree to the rounding that a
different multiply-add contraction may leave (float32 directions of a
converged solve: below 1e-9 of each array's largest entry).  Sizes: every
number of cells per lane and its edges, one stage to more stages than warps,
single instances (clusters for long horizons) and batches, several actuators
on a lane and on a cell, warm and shifted starts, the iteration limit, and a
state that diverges."""
import numpy as np
import pytest

from paper_2004_02484_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2004_02484_gb300 import build as b
    b.build()
    import torch
    torch.cuda.set_device(0)
    from paper_2004_02484_gb300 import nmpc as G
    return G


def _solve(G, insts, graph, inits=(0,), **opts):
    import torch
    s = G.Solver(insts, precision=G.NMPC_MIXED, use_graph=graph, **opts)
    assert G.nmpc_line_plan(s.h)["instances"] == len(insts)
    out = []
    for init in inits:
        rc, st = s.solve(init=init)
        torch.cuda.synchronize()
        out.append((rc, [(x.iters, x.status, x.f64_iters) for x in st],
                    np.array([[x.res_inf, x.res_2] for x in st]),
                    [t.cpu().numpy() for t in s.state()]))
    s.close()
    return out


def _same(a, b, rtol=1e-9):
    for (rc, st, res, state), (rc2, st2, res2, state2) in zip(a, b):
        assert rc == rc2 and st == st2
        assert np.allclose(res, res2, rtol=1e-4, equal_nan=True)
        for x, y in zip(state, state2):
            assert np.abs(x - y).max() <= rtol * max(np.abs(y).max(), 1e-300)


@pytest.mark.parametrize("m,n,nu", [(1, 1, 1), (7, 3, 1), (32, 20, 2), (33, 2, 1), (64, 17, 2), (65, 33, 3),
                                    (96, 16, 4), (97, 10, 2), (128, 21, 4), (129, 50, 3), (160, 8, 1),
                                    (193, 31, 2), (225, 60, 4), (256, 60, 4)])
def test_single_instances(G, m, n, nu):
    insts = [wl.heat1d(m, n, nu, 0.01, seed=11 + m)]
    kw = dict(tol=1e-6, max_iter=4000)
    _same(_solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw))


@pytest.mark.parametrize("n_lo,n_u_it", [(1, 1), (2, 1), (3, 2)])
def test_ragged_batch(G, n_lo, n_u_it):
    insts = wl.heat1d_ragged_batch(n=150, base_seed=8000)
    kw = dict(tol=1e-6, max_iter=4000, n_lo=n_lo, n_u_it=n_u_it)
    _same(_solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw))


def test_actuators_on_a_lane_and_on_a_cell(G):
    insts = [wl.heat1d(200, 12, 6, 0.01, seed=5, act_pos=[0.2, 0.2, 0.205, 0.21, 0.8, 0.99]),
             wl.heat1d(40, 9, 64, 0.01, seed=6, act_pos=[(a + 1) / 65 for a in range(64)])]
    for n_u_it in (1, 2):
        kw = dict(tol=1e-6, max_iter=400, n_u_it=n_u_it)
        _same(_solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw))


def test_warm_and_shifted_starts(G):
    insts = wl.heat1d_ragged_batch(n=6, base_seed=8200)
    kw = dict(tol=1e-7, max_iter=4000)
    inits = (G.NMPC_INIT_COLD, G.NMPC_INIT_WARM, G.NMPC_INIT_SHIFT)
    a, b = _solve(G, insts, 1, inits, **kw), _solve(G, insts, 0, inits, **kw)
    _same(a, b)
    assert all(it == 0 for it, _, _ in a[1][1])  # an already converged state returns at once


@pytest.mark.parametrize("max_iter", [0, 1, 17])
def test_iteration_limit(G, max_iter):
    insts = wl.heat1d_ragged_batch(n=5, base_seed=8300)
    kw = dict(tol=1e-9, max_iter=max_iter)
    a, b = _solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw)
    _same(a, b, rtol=1e-6)
    assert a[0][0] == G.NMPC_ERR_NOT_CONVERGED


def test_a_diverging_instance_returns_what_the_iterations_return(G):
    insts = wl.heat1d_ragged_batch(n=3, base_seed=8400)
    insts[1].x0 = insts[1].x0.copy()
    insts[1].x0[3] = np.nan
    kw = dict(tol=1e-6, max_iter=2000)
    (a,), (b,) = _solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw)
    assert a[0] == b[0] == G.NMPC_ERR_DIVERGED and a[1] == b[1]
    for x, y in zip(a[3], b[3]):
        assert np.array_equal(np.isnan(x), np.isnan(y))
        ok = ~np.isnan(y)
        assert np.abs(x[ok] - y[ok]).max() <= 1e-9 * np.abs(y[ok]).max()


@pytest.mark.parametrize("init", ["cold", "shift"])
def test_only_the_diverging_instance_is_iterated(G, init):
    """One start state with a NaN among 24: that instance alone goes through the
    iterations (it stops in their first chunk), the others keep the solutions
    of the whole-instance launches, bit for bit those of a batch without it."""
    import torch
    insts = wl.heat1d_ragged_batch(n=24, base_seed=8500)
    bad, out = 7, []
    for with_nan in (False, True):
        s = G.Solver(insts, precision=G.NMPC_MIXED, tol=1e-6, max_iter=2000)
        if init == "shift":
            assert s.solve()[0] == G.NMPC_OK
        if with_nan:
            s.x0[sum(i.mx for i in insts[:bad]) + 3] = float("nan")
        before = G.nmpc_launch_plan(s.h)["iteration_launches"]
        rc, st = s.solve(init=G.NMPC_INIT_COLD if init == "cold" else G.NMPC_INIT_SHIFT)
        launches = G.nmpc_launch_plan(s.h)["iteration_launches"] - before
        assert launches == (1 + 16 if with_nan else 1)  # the default check_every
        assert [e.status for e in st] == [G.NMPC_STATUS_DIVERGED if with_nan and b == bad
                                          else G.NMPC_STATUS_CONVERGED for b in range(s.n)]
        x, u, lam = s.state()
        out.append((torch.split(x, [i.horizon * i.mx for i in insts]),
                    torch.split(u, [i.horizon * len(i.act) for i in insts]),
                    torch.split(lam, [i.horizon * i.mx for i in insts]), [e.iters for e in st]))
        s.close()
    for b in range(len(insts)):
        if b != bad:
            assert all(torch.equal(out[0][q][b], out[1][q][b]) for q in range(3))
            assert out[0][3][b] == out[1][3][b]


# (cells, N, instances, whole-instance launches): every cells-per-lane form as
# clusters of eight, four and two CTAs or one, with as many warps as stages or
# batch form; long horizons and batches whose CTAs would leave SMs idle stay on
# launches by iteration
ROUTES = [(32, 60, 1, True), (64, 64, 1, True), (128, 33, 4, True), (256, 60, 4, True), (256, 60, 20, True),
          (128, 40, 36, True), (32, 110, 44, True), (256, 60, 44, True), (64, 20, 100, True),
          (128, 110, 28, True), (256, 60, 100, True), (32, 66, 1, False), (64, 80, 4, False),
          (128, 110, 12, False), (32, 160, 20, False), (256, 160, 4, False), (256, 40, 44, False),
          (256, 66, 76, False), (256, 65, 40, False), (256, 40, 76, False)]


@pytest.mark.parametrize("m,n,k,whole", ROUTES)
def test_route(G, m, n, k, whole):
    insts = [wl.heat1d(m, n, 2, 0.01, seed=40 + b) for b in range(k)]
    kw = dict(tol=1e-5, max_iter=2000)
    s = G.Solver(insts, precision=G.NMPC_MIXED, **kw)
    before = G.nmpc_launch_plan(s.h)["iteration_launches"]
    assert s.solve()[0] == G.NMPC_OK
    launches = G.nmpc_launch_plan(s.h)["iteration_launches"] - before
    s.close()
    assert (launches == 1) == whole
    _same(_solve(G, insts, 1, **kw), _solve(G, insts, 0, **kw))
