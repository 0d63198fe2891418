"""The batched Hines solve where a block's chain tables overflow before the
block has seen an invalid tree of its own: the invalid tree is rejected, and
the block's other trees are solved once -- also where the output is the rhs, so
that a second solve would take the solution as its rhs -- through both entry
points and on two calls in a row."""
import numpy as np
import pytest

import oracle
from paper_2005_06332_gb300 import mm, netgen

pytestmark = pytest.mark.gpu


def test_trees_beside_an_invalid_one_are_solved_once():
    import torch
    star = np.concatenate([[-1], np.zeros(1598, np.int64), [-7]])  # 1,598 chains, then an entry without a parent
    rng = np.random.default_rng(2)
    # blocks of two trees (mean size 500 of a million entries): an invalid and a valid one
    trees = [t for k in range(300) for t in (star, netgen.random_tree(rng, 100, 0.2))]
    trees += [netgen.random_tree(rng, 350, 0.1) for _ in range(1400)]
    off = np.concatenate([[0], np.cumsum([len(t) for t in trees])]).astype(np.int64)
    n = int(off[-1])
    par = np.concatenate(trees).astype(np.int32)
    a, c = -rng.uniform(0.1, 1.0, n), -rng.uniform(0.1, 1.0, n)
    b, r = rng.uniform(30.0, 40.0, n), rng.normal(size=n)
    dev = [torch.as_tensor(v, device="cuda") for v in (off, par, a, b, c)]
    L = mm.load()
    good = [k for k in range(len(trees)) if len(trees[k]) != 1600]
    ref = {k: oracle.hines_solve(*(v[off[k]:off[k + 1]] for v in (a, b, c, r)), trees[k].astype(np.int32)) for k in good}
    for fn in (L.mm_hines_solve, L.mm_hines_solve_noalloc, L.mm_hines_solve_noalloc):
        x = torch.as_tensor(r, device="cuda").clone()
        assert fn(len(trees), n, *(v.data_ptr() for v in dev), x.data_ptr(), x.data_ptr(),
                  torch.cuda.current_stream().cuda_stream) == mm.MM_EINVAL
        got = x.cpu().numpy()
        for k in good:
            np.testing.assert_allclose(got[off[k]:off[k + 1]], ref[k], rtol=1e-12, atol=1e-14)


def test_large_trees_of_one_block_match_algorithm_1():
    """Large bushy trees before many tiny ones: several fall into one block, whose tables hold the chains of none."""
    import torch
    rng = np.random.default_rng(6)
    trees = [netgen.random_tree(rng, 9000 + 500 * k, 0.6) for k in range(7)]
    trees += [netgen.random_tree(rng, 1 + k % 60, 0.2) for k in range(20000)]
    off = np.concatenate([[0], np.cumsum([len(t) for t in trees])]).astype(np.int64)
    n = int(off[-1])
    a, c = -rng.uniform(0.1, 1.0, n), -rng.uniform(0.1, 1.0, n)
    kids = np.concatenate([np.bincount(t[1:], minlength=len(t)) for t in trees])
    b, r = rng.uniform(1.5, 3.0, n) + 1.5 * kids, rng.normal(size=n)
    x = mm.hines_solve(*(torch.as_tensor(v, device="cuda")
                         for v in (off, np.concatenate(trees).astype(np.int32), a, b, c, r))).cpu().numpy()
    ref = [oracle.hines_solve(*(v[s:e] for v in (a, b, c, r)), t.astype(np.int32)) for s, e, t in zip(off[:-1], off[1:], trees)]
    np.testing.assert_allclose(x, np.concatenate(ref), rtol=1e-12, atol=1e-14)


@pytest.mark.parametrize("sizes", [[1], [8], [7, 8, 0, 1], [8, 9], [1, 8, 24], [8, 2000]])
def test_tiny_trees_match_algorithm_1(sizes):
    """Blocks of trees of up to eight entries (a thread solves each), and of one more, empty trees and large ones among them."""
    import torch
    rng = np.random.default_rng(8)
    trees = [netgen.random_tree(rng, sizes[k % len(sizes)], 0.3) if sizes[k % len(sizes)] else np.zeros(0, np.int32)
             for k in range(1000)]
    off = np.concatenate([[0], np.cumsum([len(t) for t in trees])]).astype(np.int64)
    n = int(off[-1])
    a, c = -rng.uniform(0.1, 1.0, n), -rng.uniform(0.1, 1.0, n)
    b, r = rng.uniform(8.0, 9.0, n), rng.normal(size=n)
    x = mm.hines_solve(*(torch.as_tensor(v, device="cuda")
                         for v in (off, np.concatenate(trees).astype(np.int32), a, b, c, r))).cpu().numpy()
    for s, e, t in zip(off[:-1], off[1:], trees):
        if e > s:
            np.testing.assert_allclose(x[s:e], oracle.hines_solve(*(v[s:e] for v in (a, b, c, r)), t.astype(np.int32)),
                                       rtol=1e-12, atol=1e-14)


@pytest.mark.parametrize("count,n,step", [(4000, 1000, 2), (1200, 1500, 1), (160, 8300, 1), (3, 700, 1)])
def test_deep_trees_match_algorithm_1(count, n, step):
    """Combs (step 1: two spines, every entry a chain; step 2: a spine whose entries have a leaf each, in preorder), whose
    levels are as many as half their entries: more blocks than the chip holds at a time, larger than the tables, and few."""
    import torch
    rng = np.random.default_rng(7)
    i = np.arange(n)
    par = np.maximum(i - 2, 0) if step == 1 else np.where(i % 2 == 1, i - 1, np.maximum(i - 2, 0))
    par[0] = -1
    off = np.arange(count + 1, dtype=np.int64) * n
    N = count * n
    a, c, r = -rng.uniform(0.1, 1.0, N), -rng.uniform(0.1, 1.0, N), rng.normal(size=N)
    b = rng.uniform(4.0, 5.0, N)
    x = mm.hines_solve(*(torch.as_tensor(v, device="cuda")
                         for v in (off, np.tile(par, count).astype(np.int32), a, b, c, r))).cpu().numpy()
    for s in range(0, N, max(n, N // 40 // n * n)):  # forty of them
        e = s + n
        np.testing.assert_allclose(x[s:e], oracle.hines_solve(a[s:e], b[s:e], c[s:e], r[s:e], par.astype(np.int32)),
                                   rtol=1e-12, atol=1e-14)
