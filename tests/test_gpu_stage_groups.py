"""The plate and wave direction kernels at the edges of their thread groups:
one and two points per thread (256 / 257 points), groups of a whole warp and
one point more, several stages per thread block, every sweep count's exchange
pattern (n_lo = 1, 2, 3) and no u-iteration.  One iteration against the
oracles' float64 one: 1e-11 of each field's largest entry (the same terms in
another order: a few ulps)."""
import numpy as np
import pytest

from oracle import plate as P
from oracle import wave as Wv
from paper_2004_02484_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

WAVES = {
    "string_32": lambda: [wl.wave_instance(m=32, horizon=3, T=0.009)],
    "string_33_neumann": lambda: [wl.wave_instance(m=33, horizon=3, T=0.009, bc="neumann")],
    "string_257": lambda: [wl.wave_instance(m=257, horizon=2, T=2e-5)],
    "membrane_16": lambda: [wl.wave_instance(dim=2, m=16, horizon=3, T=0.009)],
    "membrane_17_neumann": lambda: [wl.wave_instance(dim=2, m=17, horizon=3, T=0.009, bc="neumann")],
    "membrane_32": lambda: [wl.wave_instance(dim=2, m=32, horizon=2, T=0.006, n_act=3)],
    "shared_blocks": lambda: [wl.wave_instance(m=20 + (b % 3), horizon=13, T=0.039, seed=b)
                              for b in range(50)],
}
PLATES = {
    "plate_5x5": lambda: [wl.plate_instance(m=5, horizon=3, T=15.0, act_idx=(1, 3))],
    "plate_16x16": lambda: [wl.plate_instance(m=16, horizon=2, T=10.0)],
    "plate_17x17": lambda: [wl.plate_instance(m=17, horizon=3, T=15.0)],
    "plate_32x32": lambda: [wl.plate_instance(m=32, horizon=2, T=2.0)],
    "line_dirichlet_33": lambda: [wl.pinned_heat1d(m=33, horizon=4, h=1e-3, r=1.0)],
    "shared_blocks": lambda: wl.plate_batch(41, m=7, horizon=15, act_idx=(1, 4)),
}
SWEEPS = [(1, 2), (2, 0), (2, 2), (3, 1)]


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _check(solver, probs, states, oracle_step, check):
    pk = lambda A: np.concatenate([a.reshape(-1) for a in A])
    (xo, uo, lo), _ = solver.iterate(*(_t(pk([st[q] for st in states])) for q in range(3)), 1)
    got = [t.cpu().numpy() for t in (xo, uo, lo)]
    solver.close()
    at = [0, 0, 0]
    for b, p in enumerate(probs):
        want = oracle_step(p, *states[b])
        for q in range(3):
            n = want[q].size
            if b in check:
                g = got[q][at[q]:at[q] + n].reshape(want[q].shape)
                assert np.abs(g - want[q]).max() <= 1e-11 * np.abs(want[q]).max(), (b, q)
            at[q] += n


@pytest.mark.parametrize("n_lo,n_u_it", SWEEPS)
@pytest.mark.parametrize("variant,name", [(0, "jacobi"), (1, "redblack")])
@pytest.mark.parametrize("case", list(WAVES))
def test_wave_iteration(case, variant, name, n_lo, n_u_it):
    from paper_2004_02484_gb300 import wave as GW
    insts = WAVES[case]()
    probs = [Wv.WaveProblem(i) for i in insts]
    rng = np.random.default_rng(5)
    states = []
    for p in probs:
        X, U, L = p.cold_start()
        states.append((X + 0.05 * rng.standard_normal(X.shape), U + 0.5 * rng.standard_normal(U.shape),
                       L + 0.01 * rng.standard_normal(L.shape)))
    _check(GW.WaveSolver(insts, variant=variant, n_lo=n_lo, n_u_it=n_u_it), probs, states,
           lambda p, X, U, L: Wv.iteration(p, X, U, L, name, n_lo, n_u_it)[:3],
           {0, len(insts) // 2, len(insts) - 1})


@pytest.mark.parametrize("n_lo,n_u_it", SWEEPS)
@pytest.mark.parametrize("variant,name", [(0, "jacobi"), (1, "redblack")])
@pytest.mark.parametrize("case", list(PLATES))
def test_plate_iteration(case, variant, name, n_lo, n_u_it):
    from paper_2004_02484_gb300 import plate as GP
    insts = PLATES[case]()
    probs = [P.PinnedProblem(i) for i in insts]
    rng = np.random.default_rng(6)
    states = []
    for p in probs:
        X, U, L = p.cold_start()
        wide = p.tau > 0
        X = X + (15.0 if wide else 0.05) * rng.standard_normal(X.shape)
        U = rng.uniform(p.u_lo + 20, p.u_hi - 20, U.shape) if wide else U + 0.3 * rng.standard_normal(U.shape)
        states.append((X, U, L + 1e-3 * rng.standard_normal(L.shape)))
    _check(GP.PlateSolver(insts, variant=variant, n_lo=n_lo, n_u_it=n_u_it), probs, states,
           lambda p, X, U, L: P.iteration(p, X, U, L, name, n_lo, n_u_it)[:3],
           {0, len(insts) // 2, len(insts) - 1})


# one stage kind with grids of both thread shapes, more of them than run at once
MIXED_WAVES = lambda: ([wl.wave_instance(dim=2, m=5, horizon=5, T=0.015, seed=b) for b in range(70)] +
                       [wl.wave_instance(dim=2, m=17, horizon=3, T=0.009)])
MIXED_PLATES = lambda: wl.plate_batch(45, m=5, horizon=7, act_idx=(1, 3)) + [wl.plate_instance(m=17, horizon=3, T=15.0)]


@pytest.mark.parametrize("variant,name", [(0, "jacobi"), (1, "redblack")])
def test_grids_of_both_thread_shapes(variant, name):
    from paper_2004_02484_gb300 import plate as GP
    from paper_2004_02484_gb300 import wave as GW
    rng = np.random.default_rng(7)
    insts = MIXED_WAVES()
    probs = [Wv.WaveProblem(i) for i in insts]
    states = []
    for p in probs:
        X, U, L = p.cold_start()
        states.append((X + 0.05 * rng.standard_normal(X.shape), U + 0.5 * rng.standard_normal(U.shape),
                       L + 0.01 * rng.standard_normal(L.shape)))
    _check(GW.WaveSolver(insts, variant=variant), probs, states,
           lambda p, X, U, L: Wv.iteration(p, X, U, L, name, 2, 2)[:3], {0, 40, 69, 70})
    insts = MIXED_PLATES()
    probs = [P.PinnedProblem(i) for i in insts]
    states = []
    for p in probs:
        X, U, L = p.cold_start()
        states.append((X + 15.0 * rng.standard_normal(X.shape), rng.uniform(p.u_lo + 20, p.u_hi - 20, U.shape),
                       L + 1e-3 * rng.standard_normal(L.shape)))
    _check(GP.PlateSolver(insts, variant=variant), probs, states,
           lambda p, X, U, L: P.iteration(p, X, U, L, name, 2, 2)[:3], {0, 22, 44, 45})
