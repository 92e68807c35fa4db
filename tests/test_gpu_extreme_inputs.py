"""FP64 calls at the ends of what the handles accept: sample totals so small
that their reciprocal overflows, branches of nearly the largest FP64 value, and
more jobs in a call than 65,535 blocks of 32 plane rows hold."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import Table as STable, table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]


@pytest.fixture(autouse=True)
def options():
    yield
    uf.uf_set_option("sparse", 1)
    uf.uf_set_option("tensor_path", 1)


def check(tree_s, table_s, methods, what, sparse=(0, 1)):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    for method in methods:
        alpha = 0.5 if method == "generalized" else 1.0
        exp = oracle.condensed(tree_s, table_s, method, alpha)
        assert np.isfinite(exp).all()
        for s in sparse:
            uf.uf_set_option("sparse", s)
            got, _ = uf.uf_compute(tree, table, method, alpha, "fp64")
            assert_close(got, exp, method, "fp64", f"{what} sparse={s}")
        if method in ("unweighted", "weighted_normalized", "weighted_unnormalized", "generalized"):
            out = torch.full((exp.size,), -1.0, dtype=torch.float64, device="cuda")
            uf.uf_compute_noalloc(tree, table, method, alpha, "fp64", out=out)
            assert_close(out.cpu().numpy(), exp, method, "fp64", f"{what} allocation-free")


@pytest.mark.parametrize("n", [20, 50])
@pytest.mark.parametrize("count", [1e-320, 1e-310, 1e-300, 1e300, 1e306])
def test_counts_of_any_magnitude(n, count):
    tree_s = yule_tree(120, seed=2300)
    table_s = table_iid(n, 120, 0.1, seed=2301)
    # two samples of this magnitude among ordinary ones; integer multiples of it sum exactly
    for k in (3, n - 1):
        a, b = table_s.indptr[k], table_s.indptr[k + 1]
        table_s.data[a:b] = count * np.minimum(table_s.data[a:b], 8.0)
    check(tree_s, table_s, ["weighted_normalized", "weighted_unnormalized", "generalized", "unweighted"],
          f"n={n} counts of {count:g}")


@pytest.mark.parametrize("n", [20, 50])
@pytest.mark.parametrize("tensor", [0, 1])
def test_a_branch_of_any_length_that_no_sample_has(n, tensor):
    tree_s = yule_tree(120, seed=2310)
    tree_s.length *= 1e-4
    tips = np.setdiff1d(np.arange(tree_s.n_nodes), tree_s.parent)
    counts = table_iid(n, 120, 0.1, seed=2311).dense()
    counts[:, 60] = 0.0
    counts[counts.sum(1) == 0, 0] = 1.0
    tree_s.length[tips[60]] = 1.5e308
    uf.uf_set_option("tensor_path", tensor)
    check(tree_s, STable.from_dense(counts), ["weighted_normalized", "weighted_unnormalized", "unweighted"],
          f"n={n} absent branch of 1.5e308")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_jobs_on_the_tensor_cores(precision):
    tree_s = yule_tree(40, seed=2320)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    tables, exp = [], []
    for s in range(3):
        t = table_iid(2 + s, 40, 0.3, seed=2321 + s)
        tables.append(uf.Table(t.indptr, t.indices, t.data, tree))
        exp.append(oracle.condensed(tree_s, t, "unweighted"))
    jobs = [(tables[q % 3], 0, tables[q % 3].n_samples // 2) for q in range(8200)]
    outs, reps = uf.uf_compute_ranges(tree, jobs, "unweighted", 1.0, precision)
    assert reps[0].path == 1
    for q in (0, 1, 2, 4095, 8191, 8192, 8197, 8198, 8199):
        assert_close(outs[q], exp[q % 3], "unweighted", precision, f"job {q}")
    for s in range(3):
        got = np.stack([np.asarray(o) for o in outs[s::3]])
        assert (got == got[0]).all()
