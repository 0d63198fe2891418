"""Work items packed under an automatic budget, and in a supplied order to the
nearest of a given one, against the oracle: sizes from one compartment to
beyond a full item, so that items end short of the budget, on it and past it,
and a bushy tree whose path tables close an item early.  1e-3 mV is the FP32c
bar, 1e-9 mV the FP64 one."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu

SIZES = [1, 4500, 2, 700, 255, 257, 3, 1500, 2048, 64, 64, 64, 64, 900, 1, 1, 31, 4096, 512, 512, 512, 512, 17, 1200]


@pytest.mark.parametrize("precision,tol", [("fp32c", 1e-3), ("fp64", 1e-9)])
@pytest.mark.parametrize("cost", [False, True])
@pytest.mark.parametrize("group_comps", [0, 1, 600, 2048, 4096])
def test_budgets_match_oracle(precision, tol, cost, group_comps):
    net = netgen.make_network(len(SIZES), size_dist=("mono", 1), syn_per_neuron=0, seed=9, stim_nA=(0.3, 0.9))
    rng = np.random.default_rng(10)
    p = rng.choice([0.02, 0.1, 0.8], len(SIZES))
    net.comp_offset = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, q) for n, q in zip(SIZES, p)])
    net.length_um = 5.0 + 15.0 * rng.random(net.n_comp)
    net.diam_um = 0.5 + 1.5 * rng.random(net.n_comp)
    ref = oracle.simulate(net, 60)
    order = rng.random(net.n_neurons).astype(np.float32) if cost else None
    with mm.Network(net, precision=precision, group_comps=group_comps, cost=order) as g:
        g.step(60)
        V = g.read_voltages()
        spikes = g.read_spikes()[0]
    assert np.max(np.abs(V - ref.V)) <= tol
    assert len(spikes) == ref.n_spikes
