"""Scattered branches of at most 32 count entries (a warp each) beside larger
ones (a CTA each): tables whose subtrees hold 1 .. 40 entries with samples that
several tips share, every fitting branch scattered, one table and a batch of
uneven ones, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import Table, yule_tree
from tests.gpu_util import METHODS, assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2005_05826_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


def table_of(n, tips, per_tip, seed):
    """per_tip[i % len] random samples hold tip i; every sample holds tip 0 or 1."""
    rng = np.random.default_rng(seed)
    counts = np.zeros((n, tips))
    for f in range(tips):
        m = min(n, per_tip[f % len(per_tip)])
        counts[rng.choice(n, size=m, replace=False), f] = rng.integers(1, 50, size=m) * 0.25
    counts[np.arange(n), np.arange(n) % 2] += 1.0
    return Table.from_dense(counts)


@pytest.mark.parametrize("n", [2, 31, 32, 33, 40, 90])
def test_small_rows(n):
    tree_s = yule_tree(60, seed=950 + n)
    sizes = (n, 7, n + 5)
    tables_s = [table_of(m, 60, (1, 2, 3, 8, 15, 16, 31, 32, 33, 40), 951 + m) for m in sizes]
    tree = uf.Tree(tree_s.parent, tree_s.length)
    tables = [uf.Table(t.indptr, t.indices, t.data, tree) for t in tables_s]
    uf.uf_set_option("sparse", 2)
    uf.uf_set_option("tensor_path", 0)
    try:
        for method in METHODS:
            for alpha in (0.5, 0.25) if method == "generalized" else (1.0,):
                exp = [oracle.condensed(tree_s, t, method, alpha) for t in tables_s]
                for precision in ("fp64", "mixed"):
                    got, rep = uf.uf_compute(tree, tables[0], method, alpha, precision)
                    assert rep.sparse_rows > 0
                    assert_close(got, exp[0], method, precision, f"one table n={n}")
                    outs, _ = uf.uf_compute_batch(tree, tables, method, alpha, precision)
                    for o, e in zip(outs, exp):
                        assert_close(o, e, method, precision, f"batch n={n}")
    finally:
        uf.uf_set_option("sparse", 1)
        uf.uf_set_option("tensor_path", 1)
