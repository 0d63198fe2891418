"""Giant items in a supplied order -- a small giant ahead of the huge ones, and
one between them -- with few and many other compartments beside them (the huge
ones solved by clusters of blocks, and by a block each), against the oracle
within the FP32c path's bar of 1e-3 mV."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p_branch", [0.01, 0.2])
@pytest.mark.parametrize("sizes", [[12000, 60000, 9900, 33000, 300, 40], [12000, 33000, 9900, 60000] + [40000] * 9 + [70]])
def test_giants_in_a_supplied_order(sizes, p_branch):
    rng = np.random.default_rng(4)
    net = netgen.make_network(len(sizes), size_dist=("mono", 1), syn_per_neuron=4, seed=9, stim_nA=(0.3, 0.9),
                              weight_uS=(0.0, 0.01))
    net.comp_offset = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in sizes])
    net.length_um = 5.0 + 15.0 * rng.random(net.n_comp)
    net.diam_um = 0.5 + 1.5 * rng.random(net.n_comp)
    net.syn_comp = (rng.random(net.n_syn) * np.asarray(sizes)[net.syn_dst]).astype(np.int32)
    ref = oracle.simulate(net, 60)
    with mm.Network(net, precision="fp32c", cost=np.arange(len(sizes), 0, -1).astype(np.float32)) as g:
        assert g.launch_info()["giant_items"] == sum(n > 9500 for n in sizes)
        g.step(60)
        V = g.read_voltages()
        spikes = g.read_spikes()[0]
    assert np.max(np.abs(V - ref.V)) <= 1e-3
    assert len(spikes) == ref.n_spikes
