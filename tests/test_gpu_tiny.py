"""The on-chip kernel for small lattices against the plane-streaming kernel
(chosen by an explicit launch shape): psi, p and the estimators' sums bit for
bit up to the order of FP64 additions."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu


def _run(L, plane, n_chains=3, n_md=4, **kw):
    N = int(np.prod(L))
    field = kw.pop("field", 0.0)
    if field:
        kw["h"] = workloads.rng(7).standard_normal(N) * field
    with pkg.IsingHMC(dim=len(L), L=L, beta=np.linspace(0.2, 0.23, n_chains), eps=0.8 / n_md, n_md=n_md,
                      n_chains=n_chains, **kw) as s:
        if plane:
            s.set_launch(*s.launch)
        s.set_state(workloads.start_psi(n_chains, N, 1.0, seed=4), 3)
        s.trajectories(1, 11)
        s.trajectories(5, 11)
        out = [s.state(w) for w in (pkg.ISING_STATE_PSI, pkg.ISING_STATE_PSI_PROPOSAL,
                                    pkg.ISING_STATE_P_END)]
        return out, s.records(), s.chain_sums()


# scalar rows and vectors, fewer items than a warp, one to four items a thread,
# planes of more than 256 items, the largest taken
@pytest.mark.parametrize("L", [(3, 3), (4, 4), (5, 7), (16, 16), (8, 23), (33, 20), (512, 4), (1000, 8),
                               (3, 3, 3), (4, 5, 6), (6, 7, 5), (16, 16, 8), (20, 16, 3)])
@pytest.mark.parametrize("kw", [
    {}, {"h": 0.04, "flip_every": 2}, {"field": 0.1, "integrator": pkg.ISING_INTEGRATOR_OMELYAN},
    {"n_md": 1, "n_chains": 1}])
def test_matches_the_plane_kernel(L, kw):
    a, b = _run(L, False, **kw), _run(L, True, **kw)
    N = int(np.prod(L))
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    assert np.array_equal(a[1][:, [1, 2, 7]], b[1][:, [1, 2, 7]])   # log u, decisions
    assert np.abs(a[1] - b[1]).max() <= 1e-12 * 6 * N   # terms of S and K are below 6 per site
    # equal partial sums, added in FP64 in another order; six trajectories
    assert np.abs(a[2] - b[2])[:, :9].max() <= 1e-12 * 6 * N
