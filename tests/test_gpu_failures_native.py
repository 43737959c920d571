"""A device error that is on the handle already when its state is set: the call
reports it and the handle's trajectory index stays."""
import pytest

import paper_1912_03278_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(dim=2, L=(16, 12)), dict(kind="infinite", n_sites=100),
    dict(dim=2, L=(6, 5), precision=pkg.ISING_PREC_PLAIN_FP64)])
@pytest.mark.parametrize("native", [True, False])
def test_device_error_leaves_the_trajectory_index(kw, native):
    import torch
    with pkg.IsingHMC(beta=0.42, eps=0.1, n_md=3, n_chains=2, **kw) as s:
        s.trajectories(3, 5)
        psi = s.state()
        bits = torch.float64 if pkg.ising_hmc_state_elem_bytes(s.h) == 8 else torch.float32
        dev = torch.from_numpy(psi).to(bits).cuda()
        pkg.ising_hmc_inject_device_error(s.h, 1)
        with pytest.raises(pkg.IsingError) as ei:
            if native:
                pkg.ising_hmc_set_state_native(s.h, dev.data_ptr(), 40)
            else:
                s.set_state(psi, 40)
        assert ei.value.status == pkg.ISING_ETIMEOUT
        assert s.traj_index == 3
