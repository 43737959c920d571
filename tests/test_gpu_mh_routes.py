"""The packed Metropolis-Hastings sweeps on each of their routes against the
oracle, bit for bit; the number of launches tells which route ran."""
import numpy as np
import pytest

import oracle
import paper_1912_03278_gb300 as pkg

pytestmark = pytest.mark.gpu


def _check(L, n_chains, calls, launches, n_therm=1, h=0.02):
    betas = np.linspace(0.3, 0.6, n_chains)
    sim = pkg.IsingMH(dim=len(L), L=L, beta=betas, h=h, n_chains=n_chains, n_therm=n_therm)
    try:
        got = []
        for n in calls:
            before = pkg.ising_mh_launch_count(sim.h)
            sim.sweeps(n, 21)
            got.append(pkg.ising_mh_launch_count(sim.h) - before)
        assert got == launches
        s, sums = sim.spins(), sim.chain_sums()
    finally:
        sim.close()
    for c in range(n_chains):
        model = oracle.Model(dim=len(L), L=L, beta=float(betas[c]), h=h, C=2 * len(L) * float(betas[c]) + 0.1)
        rs, rsums = oracle.mh_checkerboard(model, seed=21, chain=c, n=sum(calls), n_therm=n_therm)
        assert np.array_equal(s[c], rs) and np.array_equal(sums[c], rsums), c


# a cluster per chain: warps whose lanes have different numbers of words, one to
# eight CTAs
@pytest.mark.parametrize("L", [(32, 6), (96, 70), (160, 122), (64, 12, 14)])
def test_clusters(L):
    _check(L, 3, [3, 2], [1, 1])


def test_more_sweeps_than_a_launch_takes():
    _check((32, 4), 2, [4099, 4], [2, 1], n_therm=4090)


# a launch per colour: more chains than two CTAs per SM take in one wave, too few
# words to fill two; the sums alternate between two sets, the next sweep's first
# launch measures a sweep and a launch of its own the last one of a call
@pytest.mark.parametrize("calls", [[3, 2], [1, 4], [2]])
def test_a_launch_per_colour(calls):
    import torch
    n = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 6
    _check((32, 6), n, calls, [2 * k + 1 for k in calls])


@pytest.mark.parametrize("L", [(64, 4, 6), (64,)])
def test_a_launch_per_colour_in_other_dimensions(L):
    import torch
    n = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 6
    _check(L, n, [3], [7])


# more clusters than fit at once: short and long chains stay on them, those between
# take a launch per colour
@pytest.mark.parametrize("L,launches", [((64, 8), 1), ((128, 66), 7)])
def test_several_waves_of_clusters(L, launches):
    import torch
    _check(L, 4 * torch.cuda.get_device_properties(0).multi_processor_count, [3], [launches])


def test_several_waves_of_clusters_of_long_chains():
    import torch
    n = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    L, betas = (512, 512), np.linspace(0.3, 0.6, n)
    sim = pkg.IsingMH(dim=2, L=L, beta=betas, n_chains=n)
    try:
        before = pkg.ising_mh_launch_count(sim.h)
        sim.sweeps(2, 21)
        assert pkg.ising_mh_launch_count(sim.h) - before == 1
        s, sums = sim.spins(), sim.chain_sums()
    finally:
        sim.close()
    for c in (0, n - 1):
        model = oracle.Model(dim=2, L=L, beta=float(betas[c]), C=4 * float(betas[c]) + 0.1)
        rs, rsums = oracle.mh_checkerboard(model, seed=21, chain=c, n=2)
        assert np.array_equal(s[c], rs) and np.array_equal(sums[c], rsums), c


# few spins are unpacked on the host, more by a launch
@pytest.mark.parametrize("L,n_chains,launches", [((32, 6), 1, 0), ((64, 80), 32, 0), ((64, 80), 33, 1), ((128, 64), 40, 1)])
def test_spins_unpacked_on_either_side(L, n_chains, launches):
    sim = pkg.IsingMH(dim=2, L=L, beta=0.4, n_chains=n_chains)
    try:
        want = np.where(np.random.default_rng(3).random((n_chains, L[0] * L[1])) < 0.5, -1, 1).astype(np.int8)
        sim.set_spins(want, next_sweep=0)
        before = pkg.ising_mh_launch_count(sim.h)
        assert np.array_equal(sim.spins(), want)
        assert pkg.ising_mh_launch_count(sim.h) - before == launches
    finally:
        sim.close()
