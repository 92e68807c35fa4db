"""The FP64 weighted scatter in shared-memory tiles (one table of 512 to 4,096
samples): every fitting branch scattered, at sample counts around the tiles'
edges (32 and 384 samples), odd and even, against the FP64 oracle and a call of
two jobs (which scatters directly); and stripe ranges bit for bit against a call
over all of them."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import pair_subset, table_iid, yule_tree
from tests.gpu_util import assert_close, condensed_index

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

METHODS = ["weighted_normalized", "weighted_unnormalized"]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2005_05826_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


@pytest.fixture(autouse=True)
def options():
    yield
    uf.uf_set_option("sparse", 1)


def handles(tree_s, table_s):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    return tree, uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)


@pytest.mark.parametrize("n", [512, 513, 545, 767, 768, 801, 1153])
def test_tile_edges(n):
    tree_s = yule_tree(260, seed=1000 + n)
    table_s = table_iid(n, 260, 3.0 / 260, seed=1001 + n)
    tree, table = handles(tree_s, table_s)
    uf.uf_set_option("sparse", 2)
    S = n // 2
    for method in METHODS:
        exp = oracle.condensed(tree_s, table_s, method)
        got, rep = uf.uf_compute(tree, table, method, 1.0, "fp64")
        assert rep.dense_rows == 0
        assert_close(got, exp, method, "fp64", f"tiles n={n}")
        both, _ = uf.uf_compute_ranges(tree, [(table, 0, S), (table, 0, 1)], method, 1.0, "fp64")
        assert_close(got, both[0], method, "fp64", f"tiles n={n} vs the direct scatter")
        whole, _ = uf.uf_compute(tree, table, method, 1.0, "fp64", 0, S - 1)
        cuts = [0, 1, 33, S // 2, S - 40, S - 1]
        parts = [uf.uf_compute(tree, table, method, 1.0, "fp64", a, b)[0] for a, b in zip(cuts, cuts[1:])]
        np.testing.assert_array_equal(np.vstack(parts), whole)


def test_tiles_beside_dense_rows():
    tree_s = yule_tree(3000, seed=1100)
    table_s = table_iid(1300, 3000, 0.02, seed=1101)
    h = handles(tree_s, table_s)
    i, j = pair_subset(1300, 20_000, seed=12345)
    for method in METHODS:
        exp = oracle.pairs(tree_s, table_s, method, 1.0, i, j)[0]
        for sparse in (1, 2):
            uf.uf_set_option("sparse", sparse)
            got, rep = uf.uf_compute(*h, method, 1.0, "fp64")
            assert rep.sparse_rows > 0 and rep.dense_rows > 0
            assert_close(got[condensed_index(1300, i, j)], exp, method, "fp64", f"sparse={sparse}")
