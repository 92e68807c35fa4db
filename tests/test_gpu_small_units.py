"""Calls too small to fill the GPU: the small tiles (32 stripes) and the units
cut to fewer branches, every branch dense, for every method and precision at
sample counts around the small tiles' edges and with enough branches for
several units, against the FP64 oracle; and the stripes of range calls, bit
for bit those of a call over all of them (a unit's rows do not depend on the
range)."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import table_iid, yule_tree
from tests.gpu_util import METHODS, VARIANTS, assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("n,tips", [(5, 700), (33, 90), (64, 513), (67, 1200), (130, 300)])
def test_small_calls(n, tips):
    tree_s = yule_tree(tips, seed=800 + n)
    table_s = table_iid(n, tips, 0.06, seed=801 + n)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    S = n // 2
    for method in METHODS + VARIANTS:
        for alpha in (0.5, 0.3) if method == "generalized" else (1.0,):
            exp = oracle.condensed(tree_s, table_s, method, alpha)
            for precision in ("fp64", "mixed"):
                got, rep = uf.uf_compute(tree, table, method, alpha, precision)
                assert rep.sparse_rows == 0
                assert_close(got, exp, method, precision, f"n={n} tips={tips} alpha={alpha}")
                cut = max(1, S // 3)
                whole, _ = uf.uf_compute(tree, table, method, alpha, precision, 0, S - 1)
                parts = [uf.uf_compute(tree, table, method, alpha, precision, a, b)[0]
                         for a, b in ((0, cut), (cut, S - 1)) if a < b]
                if parts:
                    np.testing.assert_array_equal(np.vstack(parts), whole)
