"""The FP64 step's scaled Hines system: couplings of every size down to none at
all (uncoupled compartments), both time discretisations, synapses on paths of
all lengths up to those that a whole warp sweeps, against the oracle within
1e-9 mV (the FP64 path's bar); the FP32c path on the same networks within its
1e-3 mV."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 5, 33, 95, 97, 98, 130, 255, 1000, 3001]


def _net(p_branch, Ra, syn):
    net = netgen.make_network(len(SIZES), size_dist=("mono", 1), syn_per_neuron=syn, seed=7, stim_nA=(0.3, 0.9),
                              weight_uS=(0.0, 0.005))
    rng = np.random.default_rng(8)
    net.comp_offset = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in SIZES])
    net.length_um = 5.0 + 15.0 * rng.random(net.n_comp)
    net.diam_um = 0.5 + 1.5 * rng.random(net.n_comp)
    net.syn_comp = (rng.random(net.n_syn) * np.asarray(SIZES)[net.syn_dst]).astype(np.int32)
    if Ra is not None:
        net.params = dict(net.params, Ra=Ra)
    return net


@pytest.mark.parametrize("Ra", [None, 1e9, 1e150, 1e300, np.inf])
@pytest.mark.parametrize("scheme", ["be", "cn"])
@pytest.mark.parametrize("p_branch", [0.0, 0.1])
def test_couplings_of_every_size(p_branch, scheme, Ra):
    # less stimulus for uncoupled somata, which keep all of it (the FP32c range), and for the explicit membrane current
    net = _net(p_branch, Ra, syn=30)
    if Ra is not None or scheme == "cn":
        net.stim_nA = 1e-3 * net.stim_nA
        net.syn_w = 1e-3 * net.syn_w
    ref = oracle.simulate(net, 120, scheme=scheme)
    assert np.all(np.abs(ref.V) < 120.0)
    for precision, tol in (("fp64", 1e-9), ("fp32c", 1e-3)):
        with mm.Network(net, precision=precision, scheme=scheme) as g:
            g.step(120)
            V = g.read_voltages()
            spikes = g.read_spikes()[0]
        assert np.max(np.abs(V - ref.V)) <= tol, precision
        assert len(spikes) == ref.n_spikes, precision
