"""The batched Hines solve at the ends of FP64's range and on matrices whose
entries differ widely inside one tree: Algorithm 1's results, infinities and
NaN included, as the oracle gives them."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu


def _tree(seed, n, p=0.2):
    rng = np.random.default_rng(seed)
    par = netgen.random_tree(rng, n, p).astype(np.int32)
    a, c, r = -rng.uniform(0.1, 1.0, n), -rng.uniform(0.1, 1.0, n), rng.normal(size=n)
    return par, a, rng.uniform(1.5, 3.0, n) + 1.5 * np.bincount(par[1:], minlength=n), c, r


def _solve(trees, in_place=False):
    import torch
    off = np.concatenate([[0], np.cumsum([len(t[0]) for t in trees])]).astype(np.int64)
    dev = [torch.as_tensor(v, device="cuda") for v in (off, *(np.concatenate(v) for v in zip(*trees)))]
    if in_place:
        x = dev[5]
        assert mm.load().mm_hines_solve(len(trees), x.numel(), *(v.data_ptr() for v in dev[:5]), x.data_ptr(), x.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream) == mm.MM_OK
    else:
        x = mm.hines_solve(*dev)
    x = x.cpu().numpy()
    with np.errstate(all="ignore"):
        ref = [oracle.hines_solve(a, b, c, r, par) for par, a, b, c, r in trees]
    return [x[s:e] for s, e in zip(off[:-1], off[1:])], ref


def _same(x, ref):
    """Infinities and NaN where Algorithm 1 has them, the rest within the bound of the other shapes (their solutions are
    of size 1), scaled by the tree's largest value."""
    fine = np.isfinite(ref)
    assert np.array_equal(np.isnan(x), np.isnan(ref)) and np.array_equal(x[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)])
    np.testing.assert_allclose(x[fine], ref[fine], rtol=1e-12, atol=1e-14 * np.max(np.abs(ref[fine]), initial=0.0))


@pytest.mark.parametrize("where", ["leaf", "inside", "root", "all"])
@pytest.mark.parametrize("value", [2.0 ** 1021, 2.0 ** 1022, 1.7e308, 1e-300, 3e-308, 1e-310, 5e-324, np.inf, np.nan, 0.0, -0.0])
def test_diagonals_at_the_ends_of_the_range(value, where):
    """One diagonal (or all of a tree) at either end, but no pivots near zero, whose solutions are rounding errors; and the
    same tree scaled as a whole where the value is finite."""
    trees = []
    small = 0.0 < value < 1.0
    for seed in range(3):
        par, a, b, c, r = _tree(seed, 50)
        i = {"leaf": [49], "inside": [int(par[49])], "root": [0], "all": list(range(50))}[where]
        b[i] = value
        if not (small and where in ("leaf", "all")):
            trees.append((par, a, b, c, r))
        if 0.0 < value < 1e300 and where == "all":  # the matrix and the rhs of that size too
            _, a, b, c, r = _tree(seed, 50)
            k = min(value, 2.0 ** 1018)
            trees.append((par, a * k, b * k, c * k, r * k) if value > 1e-307 else (par, 0 * a, b * 0 + value, 0 * c, r * k))
    trees.append(_tree(9, 70))  # and a tree beside them in the block
    x, ref = _solve(trees)
    for u, v in zip(x, ref):
        _same(u, v)


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("value", [1e200, 1e308, np.inf, -np.inf, np.nan, 1e-250, 1e-310])
@pytest.mark.parametrize("k", [1, 3, 4])  # a, c, rhs
def test_rhs_and_couplings_at_the_ends_of_the_range(value, k, in_place):
    trees = []
    for seed in range(3):
        t = _tree(20 + seed, 40)
        t[k][[7, 31]] = value
        trees.append(t)
    x, ref = _solve(trees, in_place)
    for u, v in zip(x, ref):
        _same(u, v)


def test_a_roots_couplings_are_not_used():
    trees = [_tree(30 + k, 40) for k in range(4)]
    plain = _solve(trees)[0]
    for t in trees:
        t[1][0], t[3][0] = np.nan, np.inf
    for u, v in zip(_solve(trees)[0], plain):
        np.testing.assert_array_equal(u, v)


def test_a_pivot_that_cancels():
    """Leaf and root 1, couplings -1: the eliminated root is zero and the division by it infinite (NaN for a zero rhs)."""
    one = np.ones(2)
    par = np.array([-1, 0], np.int32)
    x, ref = _solve([(par, -one, one, -one, np.array(r)) for r in ([1.0, 2.0], [-3.0, 1.0], [1.0, -1.0])])
    for u, v in zip(x, ref):
        _same(u, v)


@pytest.mark.parametrize("spread", [10, 60, 90])
def test_entries_of_very_different_size_inside_one_tree(spread):
    """D A D and D rhs with D = 2^k, k drawn per entry: the solution is D^-1 that of A, within the bound of the other shapes."""
    trees, plain = [], []
    rng = np.random.default_rng(3)
    for seed, n in enumerate((2, 9, 300, 3000)):
        par, a, b, c, r = _tree(40 + seed, n, 0.1)
        k = rng.integers(-spread, spread + 1, n)
        up = k[np.maximum(par, 0)]
        trees.append((par, a * 2.0 ** (k + up), b * 2.0 ** (2 * k), c * 2.0 ** (k + up), r * 2.0 ** k))
        plain.append((oracle.hines_solve(a, b, c, r, par), 2.0 ** k))
    x, _ = _solve(trees)
    for u, (v, d) in zip(x, plain):
        np.testing.assert_allclose(u * d, v, rtol=1e-12, atol=1e-14)
