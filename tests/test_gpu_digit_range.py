"""FP64 unweighted on the tensor cores at the ends of its digits' range: longest
branches just below a power of two (whose top digit is +256), and units of
GRAM_DIGIT_KC = 16,384 branches whose digit sums reach 2^22, against the FP64
oracle and, where every length is a multiple of a power of two that both paths
hold exactly, bit for bit against the CUDA-core path."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import Table as STable, Tree as STree, table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]


def handles(tree_s, table_s):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    return tree, uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)


def compute(h, sparse, tensor):
    uf.uf_set_option("sparse", sparse)
    uf.uf_set_option("tensor_path", tensor)
    try:
        got, rep = uf.uf_compute(*h, "unweighted", 1.0, "fp64")
    finally:
        uf.uf_set_option("sparse", 1)
        uf.uf_set_option("tensor_path", 1)
    assert rep.path == tensor
    return np.asarray(got), rep


@pytest.mark.parametrize("longest", [0.998, 0.9981, 0.999, 1.999, 1.0 - 2.0 ** -40, 511.75 / 256, 1023.0 / 512,
                                     np.nextafter(2.0, 0.0), np.nextafter(2.0 ** -30, 0.0), 1.0, 2.0])
def test_longest_branch_below_a_power_of_two(longest):
    tree_s = yule_tree(60, seed=2100)
    rng = np.random.default_rng(2101)
    tree_s.length[:] = longest * rng.uniform(0.01, 0.9, size=tree_s.length.size)
    tree_s.length[rng.choice(tree_s.length.size - 1, 12, replace=False)] = longest
    table_s = table_iid(40, 60, 0.2, seed=2102)
    h = handles(tree_s, table_s)
    exp = oracle.condensed(tree_s, table_s, "unweighted")
    for sparse in (0, 1):
        assert_close(compute(h, sparse, 1)[0], exp, "unweighted", "fp64", f"longest {longest!r} sparse={sparse}")


# every digit of these multiples of 2^-62 is the same: -256 (but the top two), 255, or as drawn
SAME = {"low": sum(-256 * 512 ** t for t in range(6)) + 2 * 512 ** 6, "high": sum(255 * 512 ** t for t in range(7))}


@pytest.mark.parametrize("lengths", ["low", "high", "mixed"])
def test_longest_units(lengths):
    """A caterpillar of 20,001 tips and 2,050 samples that all hold its deepest
    tips: nearly every branch is below every sample, and the tile count gives
    units of 16,384 branches."""
    tips, n = 20_001, 2050
    # postorder: tip 0, tip 1, their parent 2, then tip and inner node in turn
    n_nodes = 2 * tips - 1
    parent = np.empty(n_nodes, dtype=np.int64)
    inner = np.arange(2, n_nodes, 2)
    parent[0] = parent[1] = 2
    parent[inner[:-1]] = inner[1:]
    parent[np.arange(3, n_nodes, 2)] = np.arange(4, n_nodes + 1, 2)
    parent[-1] = -1
    rng = np.random.default_rng(2110)
    if lengths == "mixed":  # multiples of 2^-40 up to 2: both paths hold them and their sums exactly
        length = rng.integers(1, 2 ** 41, size=n_nodes) * 2.0 ** -40
    else:
        # the nearest FP64 values: their low digits differ, the high ones and their sums stay at the ends
        length = np.full(n_nodes, SAME[lengths] * 2.0 ** -62)
    length[:-1][rng.random(n_nodes - 1) < 0.25] = 0.5
    # sample k: tips 0 and 1, and some of its own
    idx, indptr = [], [0]
    for k in range(n):
        f = np.unique(np.concatenate([[0, 1], 2 + rng.choice(tips - 2, 3, replace=False)]))
        idx.append(f)
        indptr.append(indptr[-1] + f.size)
    idx = np.concatenate(idx).astype(np.int32)
    tree_s = STree(parent, length)
    table_s = STable(n, tips, np.asarray(indptr, dtype=np.int64), idx, np.ones(idx.size))
    h = handles(tree_s, table_s)
    got, rep = compute(h, 0, 1)
    assert rep.chunk_rows == 16_384 and rep.dense_rows > 16_384
    i, j = np.triu_indices(n, k=1)
    q = rng.choice(i.size, 3000, replace=False)
    exp = oracle.pairs(tree_s, table_s, "unweighted", 1.0, i[q], j[q])[0]
    assert_close(got[q], exp, "unweighted", "fp64", f"longest units, {lengths}")
    if lengths == "mixed":
        np.testing.assert_array_equal(got, compute(h, 0, 0)[0])
