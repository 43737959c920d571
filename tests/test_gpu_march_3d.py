"""The 3D kernel that marches through the planes with register windows against
the plane-streaming kernel (chosen by an explicit launch shape): psi and p bit
for bit, energies and estimators to the rounding of their sums."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu


def _run(L, plane, split=0, n_chains=2, n_md=5, **kw):
    N = L[0] * L[1] * L[2]
    field = kw.pop("field", 0.0)
    if field:
        kw["h"] = workloads.rng(7).standard_normal(N) * field
    with pkg.IsingHMC(dim=3, L=L, beta=np.linspace(0.2, 0.23, n_chains), eps=0.8 / n_md, n_md=n_md,
                      n_chains=n_chains, **kw) as s:
        if plane:
            s.set_launch(*s.launch)
        if split:
            s.set_chain_split(split)
        s.set_state(workloads.start_psi(n_chains, N, 1.0, seed=4), 3)
        s.trajectories(1, 11)
        s.trajectories(2, 11)
        out = [s.state(w) for w in (pkg.ISING_STATE_PSI, pkg.ISING_STATE_PSI_PROPOSAL,
                                    pkg.ISING_STATE_P_END)]
        return out, s.records(), s.chain_sums()


def _same(a, b, N):
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    assert np.array_equal(a[1][:, [1, 2, 7]], b[1][:, [1, 2, 7]])   # log u, decisions
    assert np.abs(a[1] - b[1]).max() <= 1e-12 * 6 * N   # terms of S and K are below 6 per site
    # Kahan sums of four-site sums (below 4, rounded to 2.4e-7 at most each, of
    # either sign; N/4 of them) over N, three trajectories: five sigma
    assert np.abs(a[2] - b[2])[:, :9].max() <= 5 * 3 * 1.2e-7 * 0.5 / np.sqrt(N)


# one and several tiles per row, even and odd numbers of rows (one included in
# none), one warp and several, a plane of the most tiles, the fewest planes
@pytest.mark.parametrize("L", [(4, 3, 3), (4, 4, 6), (8, 5, 7), (12, 7, 16), (16, 16, 16), (24, 24, 9),
                               (20, 18, 40), (64, 64, 8), (60, 61, 5), (128, 32, 4)])
@pytest.mark.parametrize("kw", [
    {}, {"h": 0.04, "flip_every": 2}, {"field": 0.1, "integrator": pkg.ISING_INTEGRATOR_OMELYAN}])
def test_matches_the_plane_kernel(L, kw):
    _same(_run(L, False, **kw), _run(L, True, **kw), L[0] * L[1] * L[2])


@pytest.mark.parametrize("split", [2, 4, 8])
@pytest.mark.parametrize("kw", [{}, {"h": 0.04, "flip_every": 1}, {"field": 0.1}])
def test_split_chains(split, kw):
    for L in ((16, 14, 16), (8, 9, 37)):
        _same(_run(L, False, split, **kw), _run(L, True, **kw), L[0] * L[1] * L[2])


def test_falls_back_where_it_does_not_fit():
    for L in ((6, 8, 8), (32, 64, 5), (128, 33, 4)):   # ragged rows; 512 tiles; more
        try:
            a = _run(L, False)
        except pkg.IsingError:   # a plane that does not fit on chip is refused either way
            with pytest.raises(pkg.IsingError):
                _run(L, True)
            continue
        _same(a, _run(L, True), L[0] * L[1] * L[2])
