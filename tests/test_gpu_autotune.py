"""The launch-shape autotuner: memory for its temporary chains, and what it
leaves on the handle whichever kernel turns out fastest."""
import pytest

import paper_1912_03278_gb300 as pkg

pytestmark = pytest.mark.gpu


def test_falls_back_to_fewer_temporary_chains():
    import torch
    n = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    with pkg.IsingHMC(dim=2, L=(16, 16), beta=0.4, eps=0.1, n_md=3, n_chains=n) as s:
        pkg.ising_hmc_inject_alloc_failure(1)   # the first allocation of the larger temporary handle
        try:
            assert s.autotune(reps=1) > 0
        finally:
            pkg.ising_hmc_inject_alloc_failure(0)
        s.trajectories(1, 3)
        s.sync()


def test_memory_that_suffices_for_no_temporary_handle_is_reported():
    with pkg.IsingHMC(dim=2, L=(16, 16), beta=0.4, eps=0.1, n_md=3, n_chains=4) as s:
        pkg.ising_hmc_inject_alloc_failure(1)
        try:
            with pytest.raises(pkg.IsingError) as ei:
                s.autotune(reps=1)
        finally:
            pkg.ising_hmc_inject_alloc_failure(0)
        assert ei.value.status == pkg.ISING_ENOMEM


# a lattice for each kernel that can turn out fastest
@pytest.mark.parametrize("kw", [dict(dim=2, L=(16, 16), n_chains=64), dict(dim=2, L=(128, 96), n_chains=320),
                                dict(dim=3, L=(16, 16, 16), n_chains=64), dict(dim=3, L=(32, 32, 32), n_chains=160),
                                dict(dim=2, L=(1028, 24), n_chains=3)])
def test_settles_the_staging_whichever_kernel_is_fastest(kw):
    with pkg.IsingHMC(beta=0.2, eps=0.1, n_md=4, **kw) as s:
        s.autotune(reps=1)
        assert s.staging in (pkg.ISING_STAGING_THREADS, pkg.ISING_STAGING_BULK)
    with pkg.IsingHMC(beta=0.2, eps=0.1, n_md=4, **kw) as s:
        s.set_staging(pkg.ISING_STAGING_THREADS)   # a choice of the caller's stays
        s.autotune(reps=1)
        assert s.staging == pkg.ISING_STAGING_THREADS
