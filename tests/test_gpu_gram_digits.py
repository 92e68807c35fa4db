"""FP64 unweighted on the tensor cores (seven exact digits per branch length):
sample counts at tile edges, branch counts at stage and unit edges, stripe
ranges, scattered branches beside dense ones, and lengths from 1e-12 to 1e3,
against the FP64 oracle; and bit for bit against the CUDA-core path on lengths
that are multiples of 1/64, where both hold every sum exactly."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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
    uf.uf_set_option("tensor_path", 1)


def handles(tree_s, table_s):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    return tree, uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)


def compute(h, sparse, tensor, *stripes):
    uf.uf_set_option("sparse", sparse)
    uf.uf_set_option("tensor_path", tensor)
    got, rep = uf.uf_compute(*h, "unweighted", 1.0, "fp64", *stripes)
    assert rep.path == tensor
    return np.asarray(got)


@pytest.mark.parametrize("n,tips", [(2, 40), (3, 33), (127, 200), (128, 17), (129, 90), (255, 65), (257, 300),
                                    (300, 31), (520, 64), (40, 9000)])
def test_edges(n, tips):
    tree_s = yule_tree(tips, seed=900 + n)
    table_s = table_iid(n, tips, min(0.3, 20.0 / tips), seed=901 + n)
    h = handles(tree_s, table_s)
    exp = oracle.condensed(tree_s, table_s, "unweighted")
    for sparse in (0, 1, 2):
        assert_close(compute(h, sparse, 1), exp, "unweighted", "fp64", f"n={n} tips={tips} sparse={sparse}")
    S = n // 2
    if S > 2:
        whole = compute(h, 1, 1, 0, S - 1)
        parts = [compute(h, 1, 1, a, b) for a, b in ((0, 1), (1, S - 1))]
        np.testing.assert_array_equal(np.vstack(parts), whole)


def test_exact_lengths_match_the_cuda_cores_bitwise():
    tree_s = yule_tree(1500, seed=910)
    tree_s.length[:] = np.random.default_rng(911).integers(0, 500, size=tree_s.length.size) / 64.0
    table_s = table_iid(301, 1500, 0.03, seed=912)
    h = handles(tree_s, table_s)
    for sparse in (0, 1):
        np.testing.assert_array_equal(compute(h, sparse, 1), compute(h, sparse, 0))


def test_lengths_of_every_size():
    tree_s = yule_tree(400, seed=920)
    rng = np.random.default_rng(921)
    tree_s.length[:] = 10.0 ** rng.uniform(-12, 3, size=tree_s.length.size)
    tree_s.length[::13] = 0.0
    table_s = table_iid(70, 400, 0.08, seed=922)
    h = handles(tree_s, table_s)
    exp = oracle.condensed(tree_s, table_s, "unweighted")
    for sparse in (0, 1):
        assert_close(compute(h, sparse, 1), exp, "unweighted", "fp64", f"lengths 1e-12 .. 1e3 sparse={sparse}")
