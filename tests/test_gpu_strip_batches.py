"""Batches of small 2D stages on the strip path (the cluster path's split
residual, whole rows per warp up to 64 columns) against the same instances on
the cluster path (strips=2).  Given an iterate, the residual's terms are
rounded alike, so the norms of one iteration agree to the last bits; the lower
layer differs by float32 rounding: each path's direction is within 8 units in
the last place (2^-21 relative) of the exact one at its largest entry, so one
iteration's changes agree to 2^-20 of the largest.  A solve contracts those
differences with its iterates: the same count (one more or less where a norm
lands on the tolerance) and, for equal counts, solutions within 1e-8."""
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


# (mx, my, horizon, instances): the narrowest grid, 64 columns and the first
# grids of two strips, heights off the strips' rows, enough stages for strips
# and odd widths (columns copied one by one, a last pair half outside)
SIZES = [(25, 18, 9, 100), (63, 40, 20, 24), (65, 37, 25, 16), (113, 31, 24, 20), (24, 17, 7, 130), (62, 33, 20, 24), (64, 64, 50, 10), (66, 40, 30, 12), (112, 25, 20, 30),
         (114, 31, 24, 20)]


def _insts(mx, my, n, k, variant=0):
    k *= 1 + variant  # a red-black launch holds half the stages
    return [wl.heat2d(mx, my, n, 2, 2, seed=70 + b, ref_amp=0.6 + 0.01 * b) for b in range(k)]


def _solver(G, insts, strips, **opts):
    s = G.Solver(insts, precision=G.NMPC_MIXED, strips=strips, max_iter=4000, **opts)
    assert G.nmpc_strip_plan(s.h)["instances"] == (len(insts) if strips == 0 else 0)
    return s


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("variant,n_lo,n_u_it", [(0, 2, 2), (1, 2, 2), (0, 1, 1)])
def test_one_iteration_equals_the_cluster_path(G, size, variant, n_lo, n_u_it):
    import torch
    insts = _insts(*size, variant)
    gen = torch.Generator().manual_seed(3)
    out = []
    for strips in (0, 2):
        s = _solver(G, insts, strips, variant=variant, n_lo=n_lo, n_u_it=n_u_it)
        if not out:
            x0 = torch.cat([torch.from_numpy(i.x0).repeat(i.horizon) for i in insts])
            x = x0 + 0.01 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)
            lam = 1e-4 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)
            u = torch.randn(s.n_u, dtype=torch.float64, generator=gen)
            x, lam, u = x.cuda(), lam.cuda(), u.cuda()
        xo, lo, uo = torch.empty_like(x), torch.empty_like(lam), torch.empty_like(u)
        r = G.nmpc_iterate(s.h, s.x0, s.ref, x, u, lam, xo, uo, lo, 1, s.n)
        out.append((r, xo - x, uo - u, lo - lam))
        s.close()
    assert np.abs(out[0][0][:, 0] / out[1][0][:, 0] - 1).max() <= 1e-6
    for a, b in zip(out[0][1:], out[1][1:]):
        assert float((a - b).abs().max()) <= 2.0 ** -20 * float(b.abs().max())


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("variant", [0, 1])
def test_solves_follow_the_cluster_path(G, size, variant):
    insts = _insts(*size, variant)
    got = []
    for strips in (0, 2):
        s = _solver(G, insts, strips, variant=variant, tol=1e-7)
        rc, st = s.solve()
        assert rc == G.NMPC_OK
        got.append(([e.iters for e in st], [t.cpu().numpy() for t in s.state()]))
        s.close()
    it = np.array([g[0] for g in got])
    assert np.abs(it[0] - it[1]).max() <= 1
    if (it[0] == it[1]).all():
        for a, b in zip(*(g[1] for g in got)):
            assert np.abs(a - b).max() <= 1e-8 * np.abs(b).max()


def test_unaligned_iterates_are_accepted(G):
    """Stages that the cluster path would take at any alignment."""
    import torch
    insts = _insts(64, 64, 50, 3)
    s = _solver(G, insts, 0)
    n = s.n_s
    buf = torch.zeros(2 * n + 4, dtype=torch.float64, device="cuda")
    x, lam = buf[1:n + 1], buf[n + 2:2 * n + 2]
    assert x.data_ptr() % 16 == 8 or lam.data_ptr() % 16 == 8
    x.copy_(torch.cat([torch.from_numpy(i.x0).repeat(i.horizon) for i in insts]))
    u = torch.zeros(s.n_u, dtype=torch.float64, device="cuda")
    xa, la = x.clone(), lam.clone()
    assert np.array_equal(G.nmpc_residual(s.h, s.x0, s.ref, x, u, lam, s.n)[:, 0],
                          G.nmpc_residual(s.h, s.x0, s.ref, xa, u, la, s.n)[:, 0])
    outs = []
    for xi, li in ((x, lam), (xa, la)):
        o = [torch.empty_like(t) for t in (xa, u, la)]
        G.nmpc_iterate(s.h, s.x0, s.ref, xi, u, li, *o, 3, s.n)
        outs.append(o)
    assert all(torch.equal(a, b) for a, b in zip(*outs))
    s.close()


# actuators on one cell, on neighbouring cells, two cells apart
NEAR_ACTUATORS = {"one_cell": [(20, 15), (20, 15), (40, 33)],
                  "adjacent": [(20, 15), (21, 15), (40, 33), (40, 34)],
                  "two_cells": [(20, 15), (21, 16), (40, 33), (42, 33)]}


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n_lo", [1, 2])
@pytest.mark.parametrize("kind", list(NEAR_ACTUATORS))
def test_one_u_iteration_with_actuators_in_each_others_reach(G, kind, n_lo, variant):
    """n_u_it = 1: every actuator's heat counts in the rows that another one's
    control is computed from.  One iteration as on the cluster path, and solves
    that converge as its do."""
    import torch
    mx, my, n, k = 64, 50, 20, 24
    insts = _insts(mx, my, n, k, variant)
    for i in insts:
        i.act = np.asarray([y * mx + x for x, y in NEAR_ACTUATORS[kind]], dtype=np.int32)
    gen = torch.Generator().manual_seed(4)
    x0 = torch.cat([torch.from_numpy(i.x0).repeat(i.horizon) for i in insts])
    x = (x0 + 0.01 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)).cuda()
    lam = (1e-4 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)).cuda()
    u = torch.randn(sum(i.horizon * len(i.act) for i in insts), dtype=torch.float64, generator=gen).cuda()
    step, iters, status = [], [], []
    for strips in (0, 2):
        s = G.Solver(insts, precision=G.NMPC_MIXED, strips=strips, max_iter=1000, tol=1e-6,
                     variant=variant, n_lo=n_lo, n_u_it=1)
        out = [torch.empty_like(t) for t in (x, u, lam)]
        G.nmpc_iterate(s.h, s.x0, s.ref, x, u, lam, *out, 1, s.n)
        step.append([b - a for a, b in zip((x, u, lam), out)])
        st = s.solve()[1]
        iters.append(np.array([e.iters for e in st]))
        status.append([e.status for e in st])
        s.close()
    for a, b in zip(*step):
        assert float((a - b).abs().max()) <= 2.0 ** -20 * float(b.abs().max())
    assert status[0] == status[1] and np.abs(iters[0] - iters[1]).max() <= 1


@pytest.mark.parametrize("mx,my,n,k,opts,strips", [
    (64, 64, 50, 1, {}, True), (64, 64, 20, 2, {}, True), (96, 80, 5, 1, dict(variant=1), True),
    (32, 32, 20, 16, {}, True), (24, 24, 20, 192, {}, True), (64, 8, 20, 50, {}, True),
    (130, 100, 20, 2, dict(variant=1), True), (24, 90, 10, 1, {}, True),
    (64, 64, 20, 2, dict(variant=1, n_u_it=5), True),
    (64, 64, 1, 1, {}, False), (96, 80, 3, 4, {}, False), (48, 48, 20, 4, dict(variant=1), False),
    (48, 48, 20, 4, dict(n_u_it=1), False), (64, 64, 10, 1, dict(variant=1, n_u_it=1), False),
    (24, 24, 20, 64, {}, False), (24, 30, 20, 90, dict(variant=1), False),
    (32, 32, 20, 24, dict(variant=1), False)])
def test_stages_that_clusters_take_faster_stay_there(G, mx, my, n, k, opts, strips):
    s = G.Solver([wl.heat2d(mx, my, n, 2, 2, seed=b) for b in range(k)], precision=G.NMPC_MIXED, **opts)
    assert G.nmpc_strip_plan(s.h)["instances"] == (k if strips else 0)
    s.close()


@pytest.mark.parametrize("size", SIZES + [(64, 64, 50, 1), (90, 70, 20, 1)])
@pytest.mark.parametrize("n_lo", [1, 2])
def test_residual_equals_the_cluster_path(G, size, n_lo):
    """The float64 norms of one state: the same sums in another order (a few
    hundred thousand terms: 1e-12 relative)."""
    import torch
    insts = _insts(*size)
    gen = torch.Generator().manual_seed(9)
    out = []
    for strips in (0, 2):
        s = _solver(G, insts, strips, n_lo=n_lo)
        if not out:
            x0 = torch.cat([torch.from_numpy(i.x0).repeat(i.horizon) for i in insts])
            x = (x0 + 0.01 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)).cuda()
            lam = (1e-4 * torch.randn(x0.shape, dtype=torch.float64, generator=gen)).cuda()
            u = torch.randn(s.n_u, dtype=torch.float64, generator=gen).cuda()
        out.append(G.nmpc_residual(s.h, s.x0, s.ref, x, u, lam, s.n))
        s.close()
    assert np.abs(out[0] / out[1] - 1).max() <= 1e-12


def _per_instance(insts, tensors):
    cells = [i.horizon * i.mx * i.my for i in insts]
    return list(zip(*(np.split(t.cpu().numpy(), np.cumsum(n)[:-1]) for t, n in
                      zip(tensors, (cells, [i.horizon * len(i.act) for i in insts], cells)))))


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("rows", [0, 9])
def test_every_instance_of_a_mixed_batch_follows_the_cluster_path(G, rows, variant):
    """Odd and even widths, one and several strips a row, in one handle, cold and
    then shifted by a stage, also with the strips' rows given: each instance's
    count within one of the cluster path's and most of them equal, solutions
    with equal counts within 1e-8, with others within a step at the tolerance
    (1e-4 of the largest entry: the last step of a solve to 1e-7)."""
    insts = [wl.heat2d(mx, my, 20, 2, 2, seed=300 + 10 * b + q, ref_amp=0.6 + 0.01 * b)
             for b in range(10 * (1 + variant)) for q, (mx, my) in
             enumerate([(63, 65), (64, 64), (130, 40), (77, 50)])]
    sol, iters = [], []
    for strips in (0, 2):
        s = _solver(G, insts, strips, variant=variant, tol=1e-7, strip_rows=rows)
        for init in (G.NMPC_INIT_COLD, G.NMPC_INIT_SHIFT):
            rc, st = s.solve(init)
            assert rc == G.NMPC_OK
            iters.append(np.array([e.iters for e in st]))
            sol.append(_per_instance(insts, s.state()))
        s.close()
    for q in (0, 1):
        same = iters[q] == iters[q + 2]
        assert np.abs(iters[q] - iters[q + 2]).max() <= 1 and same.mean() >= 0.75
        for b in range(len(insts)):
            for x, y in zip(sol[q][b], sol[q + 2][b]):
                assert np.abs(x - y).max() <= (1e-8 if same[b] else 1e-4) * np.abs(y).max(), (q, b)
