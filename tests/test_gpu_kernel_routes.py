"""Each kernel of the FP32 lattice form on lattices where its neighbours would
take over by default, against the plane-streaming kernel; every handle is asked
which kernel it runs on.  A split of one CTA rules the on-chip kernel out, an
explicit launch shape selects the plane-streaming kernel."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads
from tests.test_gpu_parity import _parity_after, _parity_before, _parity_check, _parity_setup

pytestmark = pytest.mark.gpu

PLANE, MARCH, ONCHIP = pkg.ISING_KERNEL_PLANE, pkg.ISING_KERNEL_MARCH, pkg.ISING_KERNEL_ONCHIP
STATES = (pkg.ISING_STATE_PSI, pkg.ISING_STATE_PSI_PROPOSAL, pkg.ISING_STATE_P_END)


def _run(L, kernel, n_chains, set_start=True, **kw):
    """States and records after each of two calls (the first with the start's
    action still to be evaluated if set_start), and the sums."""
    N = int(np.prod(L))
    field = kw.pop("field", 0.0)
    if field:
        kw["h"] = workloads.rng(7).standard_normal(N) * field
    base = 0.42 if len(L) == 2 else 0.21
    with pkg.IsingHMC(dim=len(L), L=L, beta=np.linspace(base, base + 0.02, n_chains), n_chains=n_chains,
                      eps=0.8 / kw["n_md"], **kw) as s:
        if kernel == PLANE:
            s.set_launch(*s.launch)
        elif kernel == MARCH:
            s.set_chain_split(1)
        assert s.kernel == kernel
        if set_start:
            s.set_state(workloads.start_psi(n_chains, N, 1.0, seed=4), 3)
        out = []
        for n in (1, 2):
            s.trajectories(n, 11)
            out.append(([s.state(w) for w in STATES], s.records()))
        return out, s.chain_sums()


def _same(a, b, N, sums_tol, per_site):
    for (xs, ra), (ys, rb) in zip(a[0], b[0]):
        for x, y in zip(xs, ys):
            assert np.array_equal(x, y)
        assert np.array_equal(ra[:, [1, 2, 7]], rb[:, [1, 2, 7]])   # log u, decisions
        assert np.abs(ra - rb).max() <= 1e-12 * per_site * N   # terms of S and K: below per_site per site
    assert np.abs(a[1] - b[1])[:, :9].max() <= sums_tol


# Kahan FP32 sums of the same four-site terms grouped by other threads, over N:
# N/4 addends rounded to half an ulp (1.2e-7 of values around 4, of either sign), three
# trajectories, five sigma.
def _regrouped(N):
    return 5 * 3 * 1.2e-7 * 0.5 / np.sqrt(N)


# Every remainder by three of the evaluations between a trajectory's first and
# last (leapfrog n_md - 1, Omelyan 2 n_md - 1), with and without the start's
# evaluation; rows of whole vectors and ragged ones; 28 rows are too few to cut a
# chain, 97 make slabs.
@pytest.mark.parametrize("set_start", [True, False])
@pytest.mark.parametrize("rows", [28, 97])
@pytest.mark.parametrize("X", [36, 33])
@pytest.mark.parametrize("kw", [dict(n_md=n) for n in range(1, 8)] +
                         [dict(n_md=n, field=0.1, integrator=pkg.ISING_INTEGRATOR_OMELYAN) for n in (1, 2, 3)] +
                         [dict(n_md=4, h=0.04, flip_every=1)])
def test_march_2d_every_number_of_evaluations(X, rows, set_start, kw):
    L = (X, rows)
    # the sums of an uncut chain are the plane kernel's, a cut one's are regrouped
    tol = 1e-9 if rows == 28 else _regrouped(X * rows)
    _same(_run(L, MARCH, 3, set_start, **kw), _run(L, PLANE, 3, set_start, **kw), X * rows, tol, 4)


# the smallest lattices taken and one to four columns in the last thread
@pytest.mark.parametrize("L", [(4, 24), (5, 24), (7, 25), (8, 26), (32, 31), (128, 33), (3, 24)])
@pytest.mark.parametrize("kw", [dict(n_md=7), dict(n_md=6, field=0.1, integrator=pkg.ISING_INTEGRATOR_OMELYAN),
                                dict(n_md=5, h=0.04, flip_every=2)])
def test_march_2d_small_lattices(L, kw):
    _same(_run(L, MARCH, 3, **kw), _run(L, PLANE, 3, **kw), L[0] * L[1], 1e-9, 4)


@pytest.mark.parametrize("L", [(4, 3, 3), (4, 4, 6), (8, 5, 7), (12, 7, 16), (16, 16, 16), (24, 24, 9)])
@pytest.mark.parametrize("kw", [dict(n_md=1), dict(n_md=5), dict(n_md=2, field=0.1,
                                integrator=pkg.ISING_INTEGRATOR_OMELYAN), dict(n_md=4, h=0.04, flip_every=2)])
def test_march_3d_small_lattices(L, kw):
    N = int(np.prod(L))
    _same(_run(L, MARCH, 2, **kw), _run(L, PLANE, 2, **kw), N, _regrouped(N), 6)


# what each rule takes by default on few chains, and what no other kernel takes
@pytest.mark.parametrize("L,kernel", [
    ((16, 16), ONCHIP), ((64, 128), ONCHIP), ((33, 62), ONCHIP), ((16, 16, 16), ONCHIP),
    ((64, 132), MARCH), ((33, 63), MARCH), ((1024, 24), MARCH), ((32, 32, 9), MARCH),
    ((512, 20), PLANE), ((1028, 24), PLANE), ((14, 14, 14), PLANE)])
def test_default_kernels(L, kernel):
    N = int(np.prod(L))
    _same(_run(L, kernel, 2, n_md=3), _run(L, PLANE, 2, n_md=3), N, _regrouped(N), 2 * len(L))


# chains by the number (of them per SM), evaluations and field: what each rule
# leaves to the plane-streaming kernel, next to what it keeps
@pytest.mark.parametrize("L,per_sm,n_md,field,kernel", [
    ((600, 3), 1, 2, 0.0, PLANE), ((600, 3), 1, 8, 0.0, ONCHIP), ((16, 16, 8), 1, 1, 0.0, MARCH),
    ((16, 16, 8), 2, 8, 0.0, MARCH), ((16, 16, 8), 2, 8, 0.1, PLANE), ((16, 16, 16), 2, 8, 0.0, ONCHIP), ((64, 64), 2, 1, 0.0, ONCHIP),
    ((16, 16), 7, 1, 0.0, ONCHIP), ((32, 64), 7, 8, 0.0, ONCHIP), ((32, 64), 7, 2, 0.0, MARCH), ((16, 8, 8), 7, 8, 0.0, PLANE),
    ((15, 17), 7, 2, 0.0, PLANE), ((31, 33), 7, 8, 0.0, PLANE), ((31, 96), 1, 8, 0.0, MARCH), ((31, 96), 4, 8, 0.0, PLANE),
    ((61, 96), 4, 8, 0.0, MARCH), ((61, 96), 4, 8, 0.1, PLANE), ((61, 96), 7, 20, 0.0, MARCH), ((61, 96), 7, 3, 0.0, PLANE), ((99, 30), 1, 8, 0.0, PLANE),
    ((99, 30), 2, 8, 0.0, MARCH), ((255, 28), 4, 8, 0.1, MARCH), ((255, 28), 2, 8, 0.1, PLANE), ((255, 28), 8, 3, 0.1, MARCH), ((255, 28), 7, 3, 0.1, PLANE), ((301, 24), 1, 3, 0.1, PLANE),
    ((301, 24), 1, 8, 0.1, MARCH), ((128, 40), 7, 3, 0.1, PLANE), ((128, 40), 7, 3, 0.0, MARCH),
    ((16, 16, 16), 7, 8, 0.0, PLANE), ((24, 24, 24), 2, 8, 0.0, MARCH), ((24, 24, 24), 3, 8, 0.1, PLANE),
    ((16, 16, 7), 2, 8, 0.0, PLANE), ((32, 32, 16), 4, 8, 0.1, MARCH), ((32, 32, 16), 4, 2, 0.1, PLANE), ((20, 20, 20), 4, 8, 0.0, MARCH), ((20, 20, 20), 6, 8, 0.0, PLANE),
    ((32, 56, 7), 3, 8, 0.0, MARCH), ((31, 96), 3, 8, 0.0, MARCH), ((31, 96), 4, 30, 0.0, MARCH), ((31, 96), 4, 20, 0.1, PLANE)])
def test_rules(L, per_sm, n_md, field, kernel):
    import torch
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    kw = dict(h=np.full(int(np.prod(L)), field)) if field else {}
    with pkg.IsingHMC(dim=len(L), L=L, beta=0.2, eps=0.1, n_md=n_md, n_chains=n, **kw) as s:
        assert s.kernel == kernel
        s.set_chain_split(1)   # asked for: whatever takes the lattice
        assert s.kernel == (MARCH if kernel == MARCH or (len(L) == 2 and L[1] >= 24) or len(L) == 3 else PLANE)
        s.trajectories(1, 3)
        s.sync()


def test_sign_flips_count_as_shorter_trajectories():
    import torch
    n = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for flip, kernel in ((0, MARCH), (1, PLANE), (4, MARCH)):
        with pkg.IsingHMC(dim=3, L=(24, 24, 24), beta=0.2, eps=0.1, n_md=8, n_chains=n, flip_every=flip) as s:
            assert s.kernel == kernel


# many chains: several to a CTA, cut into slabs, and by default on whichever kernel pays
@pytest.mark.parametrize("n_chains", [1, 2, 320, 700])
@pytest.mark.parametrize("L,kw", [((36, 97), dict(n_md=7)), ((33, 200), dict(n_md=7, h=0.04, flip_every=2)),
                                  ((130, 49), dict(n_md=3)), ((301, 24), dict(n_md=4, field=0.1)),
                                  ((61, 48), dict(n_md=6, field=0.1, integrator=pkg.ISING_INTEGRATOR_OMELYAN))])
def test_march_2d_many_chains(L, kw, n_chains):
    _same(_run(L, MARCH, n_chains, **kw), _run(L, PLANE, n_chains, **kw), L[0] * L[1], _regrouped(L[0] * L[1]), 4)


# the chain's own configurations and decisions do not depend on the chains beside it,
# whichever kernel and split their number leads to
@pytest.mark.parametrize("L", [(64, 64), (36, 96), (33, 96), (16, 16, 16), (24, 24, 24)])
def test_chain_does_not_depend_on_its_neighbours(L):
    N = int(np.prod(L))
    base = 0.42 if len(L) == 2 else 0.21
    got, kernels = [], set()
    for n in (1, 200, 340, 1200):
        with pkg.IsingHMC(dim=len(L), L=L, beta=base, eps=0.1, n_md=8, n_chains=n) as s:
            kernels.add((s.kernel, n if s.kernel == MARCH else 0))
            s.trajectories(3, 9)
            got.append(([pkg.ising_hmc_get_chains(s.h, w, 0, 1) for w in STATES], s.records()[:1], s.chain_sums()[:1]))
    assert len(kernels) > 1
    for g in got[1:]:
        for x, y in zip(g[0], got[0][0]):
            assert np.array_equal(x, y)
        assert np.array_equal(g[1][:, [1, 2, 7]], got[0][1][:, [1, 2, 7]])
        assert np.abs(g[1] - got[0][1]).max() <= 1e-12 * 2 * len(L) * N
        assert np.abs(g[2] - got[0][2])[:, :9].max() <= _regrouped(N)


def test_other_forms_have_no_choice():
    for kw in (dict(kind="infinite", n_sites=64), dict(dim=2, L=(4, 4), precision=pkg.ISING_PREC_PLAIN_FP64)):
        with pkg.IsingHMC(beta=0.4, eps=0.1, n_md=2, **kw) as s:
            assert s.kernel == pkg.ISING_KERNEL_OTHER


# ---- the plane-streaming kernel's staging, on a launch shape of its own --------
STAGED = [
    (dict(dim=2, L=(64, 36), beta=np.array([0.44, 0.4]), h=0.02, eps=0.08, n_md=5, n_chains=2, flip_every=2), 1),
    (dict(dim=2, L=(64, 36), beta=np.array([0.44, 0.4]), h=0.02, eps=0.08, n_md=5, n_chains=2, flip_every=2), 4),
    (dict(dim=3, L=(24, 24, 16), beta=np.array([0.2217, 0.24]), h=0.05, eps=0.09, n_md=6, n_chains=2, flip_every=2), 1),
    (dict(dim=3, L=(24, 24, 16), beta=np.array([0.2217, 0.24]), h=0.05, eps=0.09, n_md=6, n_chains=2, flip_every=2), 2),
    (dict(dim=3, L=(24, 24, 16), beta=np.array([0.2217, 0.24]), h=0.05, eps=0.09, n_md=6, n_chains=2, flip_every=2), 8),
]


@pytest.mark.parametrize("kw,split", STAGED)
def test_staging_modes_of_the_plane_kernel_agree(kw, split):
    runs = []
    for mode in (pkg.ISING_STAGING_THREADS, pkg.ISING_STAGING_BULK):
        with pkg.IsingHMC(**kw) as s:
            s.set_launch(*s.launch)
            if split > 1:
                s.set_chain_split(split)
            s.set_staging(mode)
            assert s.kernel == PLANE and s.staging == mode
            s.trajectories(3, 9)
            s.trajectories(2, 9)
            runs.append([s.state(w) for w in STATES] + [s.records(), s.chain_sums()])
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("kw", [
    dict(dim=2, L=(32, 12), betas=(0.44, 0.3), h=0.05, eps=0.1, n_md=4, launch=(32, 2)),
    dict(dim=3, L=(8, 8, 8), betas=(0.22, 0.2), h=0.05, eps=0.1, n_md=4, launch=(32, 2), split=4)])
def test_bulk_staging_of_the_plane_kernel_against_the_oracle(kw):
    ctx = _parity_setup(staging=pkg.ISING_STAGING_BULK, **kw)
    try:
        assert ctx["sim"].kernel == PLANE
        _parity_before(ctx)
        ctx["sim"].trajectories(1, ctx["seed"])
    except BaseException:
        ctx["sim"].close()
        raise
    _parity_after(ctx)
    _parity_check(ctx)


def test_group_rebuilds_when_a_plane_kernel_member_changes_staging():
    def members():
        out = [pkg.IsingHMC(dim=2, L=(12, 20), beta=0.3, h=0.02, eps=0.12, n_md=4, n_chains=2),
               pkg.IsingHMC(dim=3, L=(32, 32, 8), beta=0.2217, h=0.05, eps=0.1, n_md=4, n_chains=2),
               pkg.IsingHMC(dim=2, L=(16, 16), beta=0.4, eps=0.1, n_md=6, n_chains=3)]
        for s in out[:2]:
            s.set_launch(*s.launch)
        assert [s.kernel for s in out] == [PLANE, PLANE, ONCHIP]
        return out
    ref, sw = members(), members()
    g_ref, g_sw = pkg.IsingGroup(ref), pkg.IsingGroup(sw)
    try:
        g_ref.trajectories(4, 55)
        g_sw.trajectories(2, 55)
        sw[1].set_staging(pkg.ISING_STAGING_THREADS)
        sw[0].set_staging(pkg.ISING_STAGING_BULK)
        g_sw.trajectories(1, 55)
        sw[1].set_staging(pkg.ISING_STAGING_BULK)
        g_sw.trajectories(1, 55)
        g_ref.sync()
        g_sw.sync()
        for a, b in zip(ref, sw):
            assert np.array_equal(a.state(), b.state())
            assert np.array_equal(a.chain_sums(), b.chain_sums())
    finally:
        g_ref.close()
        g_sw.close()
        for s in ref + sw:
            s.close()
