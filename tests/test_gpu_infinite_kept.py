"""Infinite-range chains too long for registers: psi and p of the leading quads
stay in shared memory, more of them when each CTA has an SM to itself.  What a
chain computes depends on neither the number kept nor the split of the calls."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu

MANY = 320   # more chains than SMs: the smaller share is kept


def _run(N, n_chains, calls, **kw):
    beta = np.linspace(0.9, 1.1, MANY)[:n_chains]
    field = kw.pop("field", 0.0)
    if field:
        kw["h"] = workloads.rng(7).standard_normal(N) * field
    with pkg.IsingHMC(kind="infinite", n_sites=N, beta=beta, eps=0.1, n_chains=n_chains, **kw) as s:
        s.set_state(workloads.start_psi(MANY, N, 1.0, seed=4)[:n_chains], 3)
        for c in calls:
            s.trajectories(c, 11)
        return [s.state(w)[:2] for w in (pkg.ISING_STATE_PSI, pkg.ISING_STATE_PSI_PROPOSAL,
                                         pkg.ISING_STATE_P_END)] + [s.records()[:2], s.chain_sums()[:2]]


# psi and p kept whole; p in part; psi whole with one CTA per SM and in part
# with two; psi in part with both; each with a last quad of 1 to 4 sites
@pytest.mark.parametrize("N", [8193, 11776, 16386, 23552, 23555, 30001, 52225, 60000])
@pytest.mark.parametrize("kw", [{"n_md": 3, "h": 0.02, "flip_every": 2}, {"n_md": 1},
                                {"n_md": 2, "field": 0.1, "integrator": pkg.ISING_INTEGRATOR_OMELYAN}])
def test_kept_share_does_not_matter(N, kw):
    a, b = _run(N, 2, [1, 1, 2], **kw), _run(N, MANY, [4], **kw)
    for x, y in zip(a, b):
        assert np.array_equal(x, y, equal_nan=True)
