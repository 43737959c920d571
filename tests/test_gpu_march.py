"""The 2D kernel that runs several force evaluations per sweep against the
plane-streaming kernel (chosen by an explicit launch shape): configurations,
proposals and momenta bit for bit, energies and estimators to the rounding of
their FP64 sums (grouped by thread, so 1e-12 of the sum)."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu


def _run(L, plane, n_chains=3, n_md=7, trajs=3, stats=True, **kw):
    N = L[0] * L[1]
    field = kw.pop("field", 0.0)
    if field:
        kw["h"] = workloads.rng(7).standard_normal(N) * field
    with pkg.IsingHMC(dim=2, L=L, beta=np.linspace(0.4, 0.46, n_chains), eps=0.9 / n_md, n_md=n_md,
                      n_chains=n_chains, **kw) as s:
        if plane:   # an explicit shape selects the plane kernel
            t, d = s.launch
            s.set_launch(t, d)
        s.set_state(workloads.start_psi(n_chains, N, 1.0, seed=4), 3)
        s.trajectories(1, 11)
        s.trajectories(trajs - 1, 11)
        out = [s.state(w) for w in (pkg.ISING_STATE_PSI, pkg.ISING_STATE_PSI_PROPOSAL,
                                    pkg.ISING_STATE_P_END)]
        return out, s.records(), s.chain_sums()


# columns: one to four in the last thread, one warp and several, a full warp;
# rows: the smallest taken and counts of every remainder by three
@pytest.mark.parametrize("L", [(4, 24), (5, 24), (7, 25), (8, 26), (32, 31), (126, 27), (128, 33),
                               (129, 24), (131, 40), (256, 64), (250, 57), (1024, 24), (1023, 25)])
@pytest.mark.parametrize("kw", [
    {}, {"h": 0.04, "flip_every": 2}, {"field": 0.1, "integrator": pkg.ISING_INTEGRATOR_OMELYAN}])
def test_matches_the_plane_kernel(L, kw):
    (a, ra, sa), (b, rb, sb) = _run(L, False, **kw), _run(L, True, **kw)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    N = L[0] * L[1]
    assert np.array_equal(ra[:, [1, 2, 7]], rb[:, [1, 2, 7]])   # log u, decisions
    assert np.abs(ra - rb).max() <= 1e-12 * 4 * N   # terms of S and K are below 4 per site
    assert np.abs(sa - sb)[:, :9].max() <= 1e-9   # means over sites of Kahan FP32 sums
    assert np.abs(sa / sb - 1)[:, 9].max() <= 1e-12 * 4 * N   # exp(-dH): relative, as dH absolute


# every remainder of the evaluations between a trajectory's first and last
@pytest.mark.parametrize("n_md", [1, 2, 3, 4, 5, 6, 8])
def test_every_number_of_steps(n_md):
    a, b = _run((36, 28), False, n_md=n_md), _run((36, 28), True, n_md=n_md)
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)


# few chains (cut into slabs of rows) and many (several to a CTA): 320 chains of
# one warp stay uncut on 152 SMs, 700 share CTAs
@pytest.mark.parametrize("n_chains", [1, 2, 320, 700])
@pytest.mark.parametrize("L,kw", [((36, 97), {}), ((33, 200), {"h": 0.04, "flip_every": 2}), ((130, 49), {}),
                                  ((64, 50), {"field": 0.1, "integrator": pkg.ISING_INTEGRATOR_OMELYAN})])
def test_slabs_and_shared_ctas(L, kw, n_chains):
    (a, ra, _), (b, rb, _) = _run(L, False, n_chains=n_chains, **kw), _run(L, True, n_chains=n_chains, **kw)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert np.array_equal(ra[:, [1, 2, 7]], rb[:, [1, 2, 7]])
    assert np.abs(ra - rb).max() <= 1e-12 * 4 * L[0] * L[1]


# warps a CTA's 256 threads do not divide into: two of 96 threads, one of 160
@pytest.mark.parametrize("n_chains", [2, 700])
@pytest.mark.parametrize("X", [300, 382, 600])
def test_uneven_groups(X, n_chains):
    a, b = _run((X, 50), False, n_chains=n_chains, n_md=4), _run((X, 50), True, n_chains=n_chains, n_md=4)
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    assert np.abs(a[1] - b[1]).max() <= 1e-12 * 4 * X * 50


@pytest.mark.parametrize("L", [(16, 16), (64, 40)])
def test_autotuned_handles_keep_their_results(L):
    out = []
    for tune in (False, True):
        with pkg.IsingHMC(dim=2, L=L, beta=0.43, eps=0.2, n_md=4, n_chains=5) as s:
            if tune:
                s.autotune(reps=1)
            s.trajectories(3, 9)
            out.append(s.state())
    assert np.array_equal(*out)


def test_falls_back_where_it_does_not_fit():
    # too few rows, rows too long: the plane kernel, same results either way
    for L in ((64, 23), (1028, 24)):
        a, b = _run(L, False), _run(L, True)
        assert all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
