"""Giant items of both kinds in one launch -- huge neurons, each solved by a
cluster of blocks, beside giants that a block solves -- and neurons of the
shared-memory classes, for chains, ordinary and bushy trees (paths around the
length from which a warp sweeps a path), against the oracle within the FP32c
path's bar of 1e-3 mV."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p_branch", [0.0, 0.05, 0.5])
@pytest.mark.parametrize("sizes,huge", [([40001, 32768, 12000, 10000, 9800, 5000, 300, 40], 2),
                                        ([32767, 10000, 9900] + [9800] * 9 + [50], 0)])
def test_huge_and_small_giants(p_branch, sizes, huge):
    rng = np.random.default_rng(4)
    net = netgen.make_network(len(sizes), size_dist=("mono", 1), syn_per_neuron=4, seed=9, stim_nA=(0.3, 0.9),
                              weight_uS=(0.0, 0.01))
    net.comp_offset = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in sizes])
    net.length_um = 5.0 + 15.0 * rng.random(net.n_comp)
    net.diam_um = 0.5 + 1.5 * rng.random(net.n_comp)
    net.syn_comp = (rng.random(net.n_syn) * np.asarray(sizes)[net.syn_dst]).astype(np.int32)
    ref = oracle.simulate(net, 120)
    with mm.Network(net, precision="fp32c") as g:
        assert g.launch_info()["giant_items"] >= huge + 3
        g.step(120)
        V = g.read_voltages()
        spikes = g.read_spikes()[0]
    assert np.max(np.abs(V - ref.V)) <= 1e-3
    assert len(spikes) == ref.n_spikes
