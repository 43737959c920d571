"""ising_hmc_get_state_native into device, pinned and pageable memory."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n_chains", [((4, 5), 1), ((5, 5), 3), ((16, 16), 700), ((7, 9), 2100)])
@pytest.mark.parametrize("where", ["device", "offset", "pinned", "pageable"])
def test_current_configurations(L, n_chains, where):
    import torch
    N = L[0] * L[1]
    with pkg.IsingHMC(dim=2, L=L, beta=0.42, eps=0.3, n_md=3, n_chains=n_chains) as s:
        s.set_state(workloads.start_psi(n_chains, N, 1.0, seed=5), 0)
        s.trajectories(2, 3)   # chains end in different buffers
        want = s.state().astype(np.float32)
        dev = "cuda" if where in ("device", "offset") else "cpu"
        buf = torch.full((n_chains * N + 2,), -7.0, device=dev, pin_memory=where == "pinned")
        out = buf[1:1 + n_chains * N] if where == "offset" else buf[:n_chains * N]   # 4-byte aligned only
        torch.cuda.synchronize()
        pkg.ising_hmc_get_state_native(s.h, out.data_ptr())
        assert np.array_equal(out.cpu().numpy().reshape(n_chains, N), want)
        guard = buf.cpu().numpy()
        assert (guard[-1] == -7.0) and (where != "offset" or guard[0] == -7.0)


def test_forms_with_one_buffer():
    import torch
    with pkg.IsingHMC(dim=2, L=(6, 5), beta=0.42, eps=0.1, n_md=3, n_chains=5,
                      precision=pkg.ISING_PREC_PLAIN_FP64) as s:
        s.trajectories(2, 3)
        out = torch.zeros((5, 30), device="cuda", dtype=torch.float64)
        torch.cuda.synchronize()
        pkg.ising_hmc_get_state_native(s.h, out.data_ptr())
        assert np.array_equal(out.cpu().numpy(), s.state())
