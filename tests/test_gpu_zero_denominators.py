"""Mixed generalized distances (alpha = 1/2) of samples whose branches all have
length 0: the denominator is 0, so the distance is.  The FP32 rows keep every
proportion at 1e-30 or more, and what that leaves in the sums is no denominator.
Short work units round those sums most often."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import Table as STable, table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]


@pytest.mark.parametrize("n,tips", [(20, 40), (64, 2000), (300, 600), (40, 9000)])
@pytest.mark.parametrize("alpha", [0.5, 0.25])
def test_samples_on_branches_of_length_0(n, tips, alpha):
    tree_s = yule_tree(tips, seed=2600)
    tip_nodes = np.setdiff1d(np.arange(tree_s.n_nodes), tree_s.parent)
    zero = np.arange(tips // 2, tips // 2 + 6)
    for v in tip_nodes[zero]:
        while tree_s.parent[v] >= 0:
            tree_s.length[v] = 0.0
            v = tree_s.parent[v]
    counts = table_iid(n, tips, max(0.02, 4.0 / tips), seed=2601).dense()
    rng = np.random.default_rng(2602)
    few = np.array([1, 5, 6, n - 1])
    counts[few] = 0.0
    counts[few[:, None], zero] = rng.integers(1, 9, size=(4, zero.size))
    table_s = STable.from_dense(counts)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    i, j = np.triu_indices(n, k=1)
    exp, _, den, _ = oracle.pairs(tree_s, table_s, "generalized", alpha, i, j)
    assert (den == 0).sum() >= 6
    try:
        for sparse in (0, 1):
            uf.uf_set_option("sparse", sparse)
            got, _ = uf.uf_compute(tree, table, "generalized", alpha, "mixed")
            assert_close(got, exp, "generalized", "mixed", f"n={n} tips={tips} alpha={alpha} sparse={sparse}")
            assert (got[den == 0] == 0).all()
    finally:
        uf.uf_set_option("sparse", 1)
    if n * tips < 100_000:
        out = torch.full((exp.size,), -1.0, dtype=torch.float64, device="cuda")
        uf.uf_compute_noalloc(tree, table, "generalized", alpha, "mixed", out=out)
        got = out.cpu().numpy()
        assert_close(got, exp, "generalized", "mixed", f"n={n} tips={tips} alpha={alpha} allocation-free")
        assert (got[den == 0] == 0).all()


@pytest.mark.parametrize("seed", range(12))
def test_small_trees_with_branches_of_length_0(seed):
    # few branches: what the floor leaves in a denominator is a few hundred grid steps
    rng = np.random.default_rng(2610 + seed)
    tips = int(rng.integers(5, 30))
    tree_s = yule_tree(tips, seed=2611 + seed)
    tree_s.length[:] = 0.25 * rng.integers(0, 5, size=tree_s.length.size) * (rng.random(tree_s.length.size) < 0.5)
    counts = np.zeros((60, tips))
    counts[np.arange(60), rng.integers(0, tips, size=60)] = rng.integers(1, 5, size=60)
    table_s = STable.from_dense(counts)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    i, j = np.triu_indices(60, k=1)
    exp, _, den, _ = oracle.pairs(tree_s, table_s, "generalized", 0.5, i, j)
    for sparse in (0, 1):
        uf.uf_set_option("sparse", sparse)
        try:
            got, _ = uf.uf_compute(tree, table, "generalized", 0.5, "mixed")
        finally:
            uf.uf_set_option("sparse", 1)
        assert_close(got, exp, "generalized", "mixed", f"seed {seed} sparse={sparse}")
        assert (got[den == 0] == 0).all()
    out = torch.full((exp.size,), -1.0, dtype=torch.float64, device="cuda")
    uf.uf_compute_noalloc(tree, table, "generalized", 0.5, "mixed", out=out)
    assert (out.cpu().numpy()[den == 0] == 0).all()
