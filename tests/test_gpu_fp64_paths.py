"""FP64 step kernel at the edges of its path sweeps: chains shorter and longer
than a sweep chunk, than the rescaling stride and than the length from which
a whole warp sweeps a path, and bushy trees whose compartments carry several
paths, against the oracle.  1e-9 mV is the FP64 path's bar."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 16, 17, 33, 94, 95, 96, 97, 98, 127, 128, 129, 161, 255, 1000, 3001]


@pytest.mark.parametrize("p_branch", [0.0, 0.05, 0.6])
@pytest.mark.parametrize("group_comps,threads", [(1, 128), (300, 256), (4096, 512)])
def test_path_lengths_match_oracle(p_branch, group_comps, threads):
    net = netgen.make_network(len(SIZES), size_dist=("mono", 1), syn_per_neuron=0, seed=7, stim_nA=(0.3, 0.9))
    rng = np.random.default_rng(8)
    net.comp_offset = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in SIZES])
    net.length_um = 5.0 + 15.0 * rng.random(net.n_comp)
    net.diam_um = 0.5 + 1.5 * rng.random(net.n_comp)
    ref = oracle.simulate(net, 120)
    with mm.Network(net, precision="fp64", group_comps=group_comps, block_threads=threads) as g:
        g.step(120)
        V = g.read_voltages()
        spikes = g.read_spikes()[0]
    assert np.max(np.abs(V - ref.V)) <= 1e-9
    assert len(spikes) == ref.n_spikes
