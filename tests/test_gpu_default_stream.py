"""Native copies are ordered after work the caller has queued on the default
stream, without a synchronise of the caller's: buffers that a kernel behind a
long one still has to write (set) or overwrite (get).  Uploads of host data are
ordered with the handle's own work however busy the default stream is."""
import numpy as np
import pytest

import paper_1912_03278_gb300 as pkg
import workloads

pytestmark = pytest.mark.gpu

KINDS = {
    "lattice": dict(dim=2, L=(32, 40), beta=0.42, eps=0.1, n_md=3, n_chains=6),
    "infinite": dict(kind="infinite", n_sites=1001, beta=0.5, eps=0.1, n_md=3, n_chains=6),
    "dense": dict(kind="dense", J=workloads.dense_couplings(128, seed=3), beta=0.3, eps=0.1, n_md=3, n_chains=6,
                  precision=pkg.ISING_PREC_BF16),
    "plain": dict(dim=2, L=(12, 10), beta=0.42, eps=0.1, n_md=3, n_chains=6, precision=pkg.ISING_PREC_PLAIN_FP64),
}


def _busy():
    import torch
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)   # about 0.1 s


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("where", ["device", "pinned"])
def test_set_state_native_waits_for_the_default_stream(kind, where):
    import torch
    with pkg.IsingHMC(**KINDS[kind]) as s:
        dt = torch.float64 if pkg.ising_hmc_state_elem_bytes(s.h) == 8 else torch.float32
        psi = torch.from_numpy(workloads.start_psi(*s.state().shape, 1.0, seed=5)).to(dt)
        want = psi.cuda()
        buf = torch.zeros(psi.shape, dtype=dt, device="cuda") if where == "device" else \
            torch.zeros(psi.shape, dtype=dt).pin_memory()
        _busy()
        buf.copy_(want, non_blocking=True)
        pkg.ising_hmc_set_state_native(s.h, buf.data_ptr(), 2)
        assert np.array_equal(s.state(), psi.double().numpy())
        assert s.traj_index == 2


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("where", ["device", "pinned"])
def test_get_state_native_waits_for_the_default_stream(kind, where):
    import torch
    with pkg.IsingHMC(**KINDS[kind]) as s:
        dt = torch.float64 if pkg.ising_hmc_state_elem_bytes(s.h) == 8 else torch.float32
        s.trajectories(2, 3)
        want = s.state()
        fill = torch.full(want.shape, -7.0, dtype=dt, device="cuda")
        buf = torch.zeros_like(fill) if where == "device" else torch.zeros(fill.shape, dtype=dt).pin_memory()
        _busy()
        buf.copy_(fill, non_blocking=True)   # has to land before the configurations
        pkg.ising_hmc_get_state_native(s.h, buf.data_ptr())
        torch.cuda.synchronize()
        assert np.array_equal(buf.cpu().double().numpy(), want)


@pytest.mark.parametrize("kind", KINDS)
def test_host_uploads_are_read_back_under_a_busy_default_stream(kind):
    with pkg.IsingHMC(**KINDS[kind]) as s:
        s.trajectories(2, 3)
        sums = s.chain_sums() + 1.0
        psi = workloads.start_psi(*s.state().shape, 1.0, seed=6)
        if kind != "plain":
            psi = psi.astype(np.float32).astype(np.float64)
        _busy()
        pkg.ising_hmc_set_sums(s.h, sums)
        assert np.array_equal(s.chain_sums(), sums)
        _busy()
        s.set_state(psi, 4)
        assert np.array_equal(s.state(), psi)
        _busy()
        pkg.ising_hmc_reset_sums(s.h)
        assert not s.chain_sums().any()
        _busy()
        pkg.ising_hmc_inject_device_error(s.h, 1)
        with pytest.raises(pkg.IsingError):
            s.sync()


@pytest.mark.parametrize("L", [(32, 8), (12, 8)])   # packed form, byte form
def test_spins_are_read_back_under_a_busy_default_stream(L):
    s = pkg.IsingMH(dim=2, L=L, beta=0.4, n_chains=3)
    try:
        spins = np.where(workloads.rng(8).random((3, L[0] * L[1])) < 0.5, -1, 1).astype(np.int8)
        _busy()
        s.set_spins(spins, next_sweep=2)
        assert np.array_equal(s.spins(), spins)
    finally:
        s.close()


def test_native_copies_under_capture_are_refused_and_leave_the_capture_usable():
    import torch
    st = torch.cuda.Stream()
    kw = dict(KINDS["lattice"], stream=st.cuda_stream)
    with pkg.IsingHMC(**kw) as a, pkg.IsingHMC(**kw) as b:
        buf = torch.zeros(a.state().shape, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for call in (lambda: pkg.ising_hmc_set_state_native(a.h, buf.data_ptr(), 0),
                         lambda: pkg.ising_hmc_get_state_native(a.h, buf.data_ptr())):
                with pytest.raises(pkg.IsingError):
                    call()
            a.trajectories(2, 7)
        with torch.cuda.stream(st):
            g.replay()
        b.trajectories(2, 7)
        torch.cuda.synchronize()
        assert np.array_equal(a.state(), b.state())
