"""The batched Hines solve over the shapes that its chain tables see: chains
around the sweep's step, stars, combs whose every entry is a chain of its own,
trees with more chains than a block's tables hold (solved by a thread each),
empty trees, tiny trees many to a block, values of very different size, a zero
pivot and an output that is the rhs itself, against the oracle's Algorithm 1."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu


def _solve(trees, scale=1.0, in_place=False, zero_pivot=None):
    import torch
    rng = np.random.default_rng(5)
    off = np.concatenate([[0], np.cumsum([len(p) for p in trees])]).astype(np.int64)
    par = np.concatenate(trees).astype(np.int32)
    n = len(par)
    a, c = -rng.uniform(0.1, 1.0, n), -rng.uniform(0.1, 1.0, n)
    kids = np.zeros(n)
    for s, e in zip(off[:-1], off[1:]):
        q = par[s:e]
        np.add.at(kids[s:e], q[1:], 1.0)
    b = rng.uniform(0.5, 2.0, n) + 1.5 * kids + 1.0
    r = rng.normal(size=n)
    k = scale ** rng.integers(-1, 2, len(trees)).repeat(np.diff(off))
    a, b, c = a * k, b * k, c * k
    if zero_pivot is not None:
        b[zero_pivot] = 0.0
    t = [torch.as_tensor(v, device="cuda") for v in (off, par, a, b, c, r)]
    if in_place:
        L = mm.load()
        x = t[5]
        assert L.mm_hines_solve(len(trees), n, *(v.data_ptr() for v in t[:5]), x.data_ptr(), x.data_ptr(),
                                torch.cuda.current_stream().cuda_stream) == mm.MM_OK
    else:
        x = mm.hines_solve(*t)
    x = x.cpu().numpy()
    with np.errstate(all="ignore"):
        ref = [oracle.hines_solve(a[s:e], b[s:e], c[s:e], r[s:e], par[s:e]) for s, e in zip(off[:-1], off[1:]) if e > s]
    return x, np.concatenate(ref)


def _chain(n):
    return np.arange(-1, n - 1)


def _star(n):
    return np.concatenate([[-1], np.zeros(n - 1, np.int64)])[:n]


def _comb(n):  # parent i - 2: no entry follows its parent, as deep as a tree of its size gets
    return np.maximum(np.arange(n) - 2, 0) - (np.arange(n) == 0)


def _random(seed, n, p):
    return netgen.random_tree(np.random.default_rng(seed), n, p)


SHAPES = {
    "chains": [_chain(n) for n in (1, 2, 3, 4, 5, 8, 9, 63, 64, 65, 1000, 5000)],
    "stars": [_star(n) for n in (1, 2, 3, 300, 4000)],
    "combs": [_comb(n) for n in (1, 2, 3, 4, 255, 2000)],
    "many_tiny": [_random(k, 1 + k % 5, 0.3) for k in range(3000)],
    "with_empty": [_random(1, 50, 0.2), np.zeros(0, np.int64), np.zeros(0, np.int64), _random(2, 7, 0.5)],
    "beyond_the_tables": [_random(3, 30, 0.2), _star(6000), _comb(9000), _random(4, 20000, 0.4), _random(5, 300, 0.1)],
    "random": [_random(10 + k, n, p) for k, (n, p) in enumerate(
        [(255, 0.1), (256, 0.1), (257, 0.1), (2047, 0.02), (2048, 0.9), (2049, 0.3), (20000, 0.05), (511, 0.5)])],
}


@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_shapes_match_algorithm_1(shape):
    x, ref = _solve(SHAPES[shape])
    np.testing.assert_allclose(x, ref, rtol=1e-12, atol=1e-14)


@pytest.mark.parametrize("scale", [1e30, 1e150])
def test_entries_of_very_different_size(scale):
    """Each tree's matrix times 1/scale, 1 or scale: the solution times the same meets the bound of the other shapes."""
    x, ref = _solve(SHAPES["random"], scale=scale)
    sizes = [len(p) for p in SHAPES["random"]]
    rng = np.random.default_rng(5)
    n = sum(sizes)
    for _ in range(2):
        rng.uniform(0.1, 1.0, n)
    rng.uniform(0.5, 2.0, n), rng.normal(size=n)
    k = scale ** rng.integers(-1, 2, len(sizes)).repeat(sizes)
    np.testing.assert_allclose(x * k, ref * k, rtol=1e-12, atol=1e-14)


def test_rhs_may_be_the_output():
    x, ref = _solve(SHAPES["random"], in_place=True)
    np.testing.assert_allclose(x, ref, rtol=1e-12, atol=1e-14)


def test_a_zero_pivot_is_no_finite_solution():
    """The leaf's diagonal is zero: the division by it spreads to the root and down the whole tree."""
    trees = [_random(1, 40, 0.2), _random(2, 60, 0.2)]
    x, ref = _solve(trees, zero_pivot=99)
    assert not np.any(np.isfinite(ref[40:]))
    np.testing.assert_allclose(x[:40], ref[:40], rtol=1e-12, atol=1e-14)
    assert not np.any(np.isfinite(x[40:]))
