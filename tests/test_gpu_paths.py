"""Passes chosen by size, storage or coefficient tables, at the sizes where the
choice or a tile changes.

 - Two-cell passes with segment words (more than 4 phases) and the FP64 pass:
   a handle that has held another state gives the bits a fresh one gives (every
   phase that is not visited must have been cleared), at segment and word edges.
 - Uniform pair coefficients (sums in registers, from constants) against the
   same problem with an extra, absent phase of other coefficients (sums from
   tables): the same terms in the same order, so the same bits.
 - Slot lists of every length up to the 12 slots (groups of four) against masked
   storage: the same bits.
 - The FP64 pass against the oracle, 1e-12 as everywhere in FP64."""
import numpy as np
import pytest

from oracle import ref
from paper_2601_16522_gb300 import inputs as I

from test_gpu_parity import REL64, pf, relerr  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

MASKED, SLOTS = 2, 16
TOL = (1e-4, 1e-2, 1e-4, 1e-3)


def _run(sim, u, integ, dt, attempts):
    sim.set_state(u)
    if attempts:
        sim.step(integ, 1e9, tol=TOL, dt0=dt, max_attempts=attempts)
    else:
        sim.step(integ, 2 * dt, dt_mult=dt / sim.dt_e())
    return sim.get_state()[0]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("nx,ny,nz,N", [(2, 5, 1, 5), (62, 9, 1, 32), (64, 6, 3, 33), (66, 5, 4, 7), (130, 7, 1, 65),
                                        (34, 9, 5, 8)])
def test_a_used_handle_equals_a_fresh_one(pf, prec, nx, ny, nz, N):
    K = N % 2
    prob, a = I.multiphase_blobs(nx, ny, nz, N, seed=1, has_conc=K, min_dist=0.6)
    b = I.multiphase_blobs(nx, ny, nz, N, seed=2, has_conc=K, min_dist=0.6)[1]
    with pf.Simulation(prob, precision=prec) as used:
        dte = used.dt_e()
        for integ, dt, attempts in [(ref.FEULER, 0.9 * dte, 0), (ref.SSP2, 2.0 * dte, 0), (ref.RKL2, 6.0 * dte, 2),
                                    (ref.RKL1, 4.0 * dte, 1)]:
            _run(used, a, integ, dt, attempts)
            got = _run(used, b, integ, dt, attempts)
            with pf.Simulation(prob, precision=prec) as fresh:
                want = _run(fresh, b, integ, dt, attempts)
            np.testing.assert_array_equal(got, want)


def _with_absent_phase(prob, u):
    """The problem and state with one more phase, present nowhere, whose pair
    coefficients differ from the others' (so the tables are not uniform)."""
    N = prob.n_phases

    def grown(m, value):
        g = np.full((N + 1, N + 1), value)
        g[:N, :N] = m
        g[N, N] = 0.0
        return g

    p2 = prob.with_(n_phases=N + 1, phase_type=np.append(prob.phase_type, prob.phase_type[-1]),
                    gamma=grown(prob.gamma, 0.5 * prob.gamma.max()),
                    mobility=grown(prob.mobility, 0.5 * prob.mobility.max()))
    return p2, np.insert(u, N, 0.0, axis=0)


@pytest.mark.parametrize("opts", [0, MASKED, SLOTS], ids=["dense", "masked", "slots"])
@pytest.mark.parametrize("nx,ny,nz,N,K,dist", [(48, 20, 1, 3, 0, None), (40, 24, 10, 9, 0, 6.0), (36, 10, 9, 31, 0, 4.0),
                                               (30, 12, 8, 8, 1, 5.0), (24, 10, 9, 12, 0, 1.5)])
def test_uniform_coefficients_equal_the_tables(pf, opts, nx, ny, nz, N, K, dist):
    # one chemical type: equal gamma and mobility for every pair
    prob, u = I.multiphase_blobs(nx, ny, nz, N, seed=4, has_conc=K, n_alpha=0, min_dist=dist)
    assert np.unique(prob.gamma[~np.eye(N, dtype=bool)]).size == 1
    p2, u2 = _with_absent_phase(prob, u)
    outs = []
    for p, v in ((prob, u), (p2, u2)):
        with pf.Simulation(p, precision=32, options=opts) as sim:
            outs.append([_run(sim, v, ref.FEULER, 0.5 * sim.dt_e(), 0), _run(sim, v, ref.RKL2, 5.0 * sim.dt_e(), 2)])
            dte = sim.dt_e()
        outs[-1].append(dte)
    assert outs[0][2] == outs[1][2]
    for one, two in zip(outs[0][:2], outs[1][:2]):
        assert not two[N].any()
        np.testing.assert_array_equal(np.delete(two, N, axis=0), one)


@pytest.mark.parametrize("n_alpha", [0, 1], ids=["uniform", "tables"])
@pytest.mark.parametrize("N", [4, 5, 8, 9, 12])
def test_slot_lists_of_every_length(pf, N, n_alpha):
    # cells of 1 to N random phases: no cell visits more than 12
    prob, _ = I.multiphase_blobs(33, 17, 5, N, seed=3, has_conc=0, n_alpha=n_alpha, min_dist=1.0)
    rng = np.random.default_rng(N)
    keep = np.argsort(np.argsort(rng.random((N, prob.V)), axis=0), axis=0) < rng.integers(1, N + 1, prob.V)
    u = np.where(keep, rng.random((N, prob.V)) + 0.05, 0.0)
    u = (u / u.sum(0)).astype(np.float32).astype(np.float64)
    res = []
    for opts in (MASKED, SLOTS):
        with pf.Simulation(prob, precision=32, options=opts) as sim:
            sim.set_state(u)
            np.testing.assert_array_equal(sim.get_state()[0], u)
            dte = sim.dt_e()
            res.append([_run(sim, u, ref.FEULER, 0.5 * dte, 0), _run(sim, u, ref.SSP2, 2.0 * dte, 0),
                        _run(sim, u, ref.RKL2, 3.0 * dte, 1)])
    for m, s in zip(*res):
        np.testing.assert_array_equal(s, m)


@pytest.mark.parametrize("nx,ny,nz,N,K", [(1, 3, 1, 3, 0), (31, 5, 1, 2, 1), (33, 9, 1, 9, 1), (64, 8, 3, 33, 0),
                                          (70, 40, 24, 3, 1), (65, 33, 40, 6, 0)])
def test_fp64_pass_against_the_oracle(pf, nx, ny, nz, N, K):
    bc = (1, 1, 0, 0, 1, 1) if K and nz > 1 else (0,) * 6
    bcc = (2, 1, 0, 0, 2, 1) if K and nz > 1 else (0,) * 6
    prob, u = I.multiphase_blobs(nx, ny, nz, N, seed=7, has_conc=K, n_alpha=1, min_dist=0.6, bc_phi=bc, bc_c=bcc,
                                 c_dirichlet=(0.6, 0, 0, 0, 0.3, 0))
    o = ref.Oracle(prob)
    dte = o.dt_e()
    with pf.Simulation(prob, precision=64) as sim:
        for integ, dt in ((ref.FEULER, 0.9 * dte), (ref.RKL2, 6.0 * dte)):
            s = 1 if integ == ref.FEULER else ref.sts_stages(integ, dt, dte)
            want, _, _, _ = o.step(integ, dt, s, u)
            sim.set_state(u)
            sim.step(integ, dt, dt_mult=dt / dte)
            assert relerr(sim.get_state()[0], want, N, K) <= REL64
