"""Host logic: work items packed under a budget chosen by the layout itself
(group_comps 0), at the edges of the choice -- one neuron, single-compartment
neurons beyond an item's neuron limit, bushy trees whose path tables would
take a full budget out of the regular class, one neuron in the large class --
checked like given budgets, and every packed item in the regular class."""
import numpy as np
import pytest

from paper_2005_06332_gb300 import netgen
from test_layout_paths import _run, checker  # noqa: F401  (fixture)

REGULAR, LARGE = 110 * 1024, 224 * 1024


@pytest.mark.parametrize("sizes,p_branch", [
    ([1], 0.0), ([4097], 0.1), ([1] * 40_000, 0.0), ([2] * 5000 + [1] * 3, 0.0),
    ([300] * 700, 0.9), ([450] * 300, 0.1), ([7000] + [37] * 500, 0.05)])
def test_chosen_budget(checker, tmp_path, sizes, p_branch):  # noqa: F811
    rng = np.random.default_rng(5)
    net = netgen.make_network(len(sizes), size_dist=("mono", 1), syn_per_neuron=0, seed=4)
    net.comp_offset = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    net.parent = np.concatenate([netgen.random_tree(rng, n, p_branch) for n in sizes])
    rc, f = _run(checker, tmp_path, net, 0, REGULAR, LARGE)
    assert rc == 0 and int(f["bad"]) == 0, f
    # only a neuron too large by itself leaves the regular class
    assert int(f["large"]) == (1 if max(sizes) > 5000 else 0) and int(f["giant"]) == 0, f
