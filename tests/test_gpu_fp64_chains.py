"""FP64 network step on long unbranched paths whose couplings are up to 7e4 times
C / dt (wide short compartments, low axial resistivity, a long time step): the
pivots of such a chain differ from the link above by little, and a sweep that
lets them cancel loses the capacitances.  Chains of all lengths around the
bounds of the warp sweep's chunks, a branched network besides.  Bars: 1e-9 mV
over 80 steps (the FP64 path's), and 2e-11 mV after the first, FP64's rounding
(1.1e-16) times the largest coupling over C / dt (7e4) times that step's dV (2.4 mV)."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu

SIZES = [4000, 1500, 700, 300, 161, 130, 129, 128, 98, 97, 96, 95, 33, 2, 1]


def _net(Ra, diam, p_branch):
    rng = np.random.default_rng(5)
    net = netgen.make_network(len(SIZES), size_dist=("mono", 1), syn_per_neuron=10, seed=6, stim_nA=(0.1, 0.6),
                              weight_uS=(0.0, 0.004), dt=0.1, delay_ms=("uniform", 0.1, 2.0))
    net.comp_offset = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in SIZES]).astype(np.int32)
    net.length_um = rng.uniform(5.0, 20.0, net.n_comp)
    net.diam_um = rng.uniform(0.5, diam, net.n_comp)
    net.syn_comp = (rng.random(net.n_syn) * np.asarray(SIZES)[net.syn_dst]).astype(np.int32)
    net.params = dict(net.params, Ra=Ra)
    net.stim_nA = net.stim_nA * np.minimum(1.0, np.asarray(SIZES) / 100.0)  # tiny neurons: within range
    return net


@pytest.mark.parametrize("scheme", ["be", "cn"])
@pytest.mark.parametrize("p_branch", [0.0, 0.02])
@pytest.mark.parametrize("Ra,diam", [(3.0, 30.0), (30.0, 30.0), (100.0, 30.0), (3.0, 2.0), (1000.0, 2.0)])
def test_strongly_coupled_chains(Ra, diam, p_branch, scheme):
    net = _net(Ra, diam, p_branch)
    if scheme == "cn":  # the explicit membrane current is stable without spikes only
        net.dt = 0.025
        net.stim_nA = 1e-3 * net.stim_nA
        net.syn_w = 1e-3 * net.syn_w
    with mm.Network(net, precision="fp64", scheme=scheme) as g:
        g.step(1)
        V1 = g.read_voltages()
        g.step(79)
        V80 = g.read_voltages()
    assert np.max(np.abs(V1 - oracle.simulate(net, 1, scheme=scheme).V)) <= 2e-11
    assert np.max(np.abs(V80 - oracle.simulate(net, 80, scheme=scheme).V)) <= 1e-9


def test_constant_roundings_do_not_add_up():
    """The diagonal's constant part is the same at every step: its rounding (up
    to 1.1e-16 of the couplings, here up to 1e4 times C / dt) must not add up over
    the steps.  18 branched neurons over 80 steps, where the oracle is within
    1.2e-14 mV (mean square) of the same steps in 80 bits; the bar is 2.5 times that."""
    rng = np.random.default_rng(101)
    sizes = np.concatenate([[4000, 1500, 700, 300, 100, 30], rng.integers(20, 400, 12)])
    net = netgen.make_network(len(sizes), size_dist=("mono", 1), syn_per_neuron=10, seed=2, stim_nA=(0.1, 0.6),
                              weight_uS=(0.0, 0.004), dt=0.025, delay_ms=("uniform", 0.1, 2.0))
    net.comp_offset = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, int(n), 0.1) for n in sizes]).astype(np.int32)
    net.length_um = rng.uniform(5.0, 20.0, net.n_comp)
    net.diam_um = rng.uniform(0.5, 2.0, net.n_comp)
    net.syn_comp = (rng.random(net.n_syn) * sizes[net.syn_dst]).astype(np.int32)
    net.params = dict(net.params, Ra=3.0)
    with mm.Network(net, precision="fp64") as g:
        g.step(80)
        V = g.read_voltages()
    assert np.sqrt(np.mean((V - oracle.simulate(net, 80).V) ** 2)) <= 3e-14
