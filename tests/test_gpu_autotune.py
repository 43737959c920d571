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
