"""The FP64 weighted and unweighted kernel on 64-bit fixed-point rows, every
branch dense (option "sparse" 0, tensor path off), against the FP64 oracle:
sample counts at the edges of its tiles, branch counts at the edges of its
pipeline stages and of its work units, and branch lengths from 1e-12 to 1e3 in
one tree.  A value is rounded to a grid of at most 2^-60 of the largest
root-to-tip distance (weighted) or of a work unit's summed lengths
(unweighted), so an entry of b branches is off by at most b 2^-61 of it: far
inside the FP64 contract for these distances."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

METHODS = ["unweighted", "unweighted_unnormalized", "weighted_normalized", "weighted_unnormalized"]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2005_05826_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


@pytest.fixture(autouse=True)
def all_dense():
    uf.uf_set_option("sparse", 0)
    uf.uf_set_option("tensor_path", 0)
    yield
    uf.uf_set_option("sparse", 1)
    uf.uf_set_option("tensor_path", 1)


def check(tree_s, table_s, what):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    for method in METHODS:
        got, rep = uf.uf_compute(tree, table, method, 1.0, "fp64")
        assert rep.sparse_rows == 0
        assert_close(got, oracle.condensed(tree_s, table_s, method), method, "fp64", what)


@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257])
def test_tile_edges(n):
    tree_s = yule_tree(60, seed=700 + n)
    check(tree_s, table_iid(n, tree_s.n_tips, 0.2, seed=701 + n), f"n={n}")


@pytest.mark.parametrize("tips", [2, 4, 5, 8, 9, 13, 33, 1024, 1025, 1030, 2100])
def test_row_edges(tips):
    tree_s = yule_tree(tips, seed=720 + tips)
    check(tree_s, table_iid(21, tips, min(1.0, max(0.05, 3.0 / tips)), seed=721 + tips), f"tips={tips}")


def test_lengths_of_every_size():
    tree_s = yule_tree(300, seed=740)
    rng = np.random.default_rng(741)
    tree_s.length[:] = 10.0 ** rng.uniform(-12, 3, size=tree_s.length.size)
    tree_s.length[::17] = 0.0
    check(tree_s, table_iid(40, 300, 0.1, seed=742), "lengths 1e-12 .. 1e3")
