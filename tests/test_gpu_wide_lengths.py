"""FP64 distances of samples whose branches are far shorter than the longest of
the tree: the contract (1e-10 relative plus 1e-15) holds for every pair, also
where other samples, or no sample, hold branches many orders of magnitude
longer.  Dense rows, scattered rows, the shared-memory tiles, the tensor cores
and the allocation-free call."""
import numpy as np
import pytest

import oracle
import paper_2005_05826_gb300 as uf
from synth import Table as STable, table_iid, yule_tree
from tests.gpu_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]

METHODS = ["unweighted", "unweighted_unnormalized", "weighted_normalized", "weighted_unnormalized"]


@pytest.fixture(autouse=True)
def options():
    yield
    uf.uf_set_option("sparse", 1)
    uf.uf_set_option("tensor_path", 1)


def check(tree_s, table_s, what, settings=((0, 1), (1, 1), (0, 0), (1, 0))):
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    n = table_s.n_samples
    for method in METHODS:
        exp = oracle.condensed(tree_s, table_s, method)
        for sparse, tensor in settings:
            uf.uf_set_option("sparse", sparse)
            uf.uf_set_option("tensor_path", tensor)
            got, rep = uf.uf_compute(tree, table, method, 1.0, "fp64")
            assert_close(got, exp, method, "fp64", f"{what} sparse={sparse} tensor={tensor}")
            assert rep.clamped == 0
        if method != "unweighted_unnormalized" and n <= 100:
            out = torch.full((exp.size,), -1.0, dtype=torch.float64, device="cuda")
            uf.uf_compute_noalloc(tree, table, method, 1.0, "fp64", out=out)
            assert_close(out.cpu().numpy(), exp, method, "fp64", f"{what} allocation-free")


def near_identical(table_s, skip, rng):
    """The table's first half followed by a variant of each sample with one count
    moved to a feature it lacks, the totals scaled to about 1e4; nobody holds
    the feature `skip`."""
    dense = table_s.dense()
    dense[:, skip] = 0.0
    half = dense.shape[0] // 2
    base = dense[:half]
    base[base.sum(1) == 0, (skip + 1) % dense.shape[1]] = 1.0
    base *= np.ceil(1e4 / base.sum(1))[:, None]
    twin = base.copy()
    for row in twin:
        free = np.setdiff1d(np.nonzero(row == 0)[0], [skip])
        row[rng.choice(np.nonzero(row)[0])] -= 1.0
        row[rng.choice(free)] += 1.0
    return np.vstack([base, twin])


@pytest.mark.parametrize("held", [False, True])
@pytest.mark.parametrize("longest", [1e3, 1e5, 1e6, 1e9, 1e13])
def test_one_long_tip(longest, held):
    tree_s = yule_tree(1000, seed=2200)
    tips = np.setdiff1d(np.arange(tree_s.n_nodes), tree_s.parent)
    f = 317
    tree_s.length[tips[f]] = longest
    counts = near_identical(table_iid(40, 1000, 0.03, seed=2201), f, np.random.default_rng(2202))
    if held:
        counts[7, f] = 1.0
    check(tree_s, STable.from_dense(counts), f"tip of {longest:g}, held by {int(held)}")


@pytest.mark.parametrize("held", [False, True])
@pytest.mark.parametrize("longest", [1e3, 1e6, 1e9])
def test_one_long_tip_scattered(longest, held):
    # 600 samples: FP64 weighted rows go through the shared-memory tiles
    tree_s = yule_tree(260, seed=2210)
    tips = np.setdiff1d(np.arange(tree_s.n_nodes), tree_s.parent)
    f = 100
    tree_s.length[tips[f]] = longest
    counts = near_identical(table_iid(600, 260, 5.0 / 260, seed=2211), f, np.random.default_rng(2212))
    if held:
        counts[7, f] = 1.0
    check(tree_s, STable.from_dense(counts), f"600 samples, tip of {longest:g}, held by {int(held)}", ((2, 1), (1, 1)))


@pytest.mark.parametrize("short", [1e-3, 1e-6, 1e-8, 1e-10, 1e-12])
def test_a_clade_of_short_branches(short):
    tips = 200
    tree_s = yule_tree(tips, seed=2220)
    # an inner node over about half of the tips: its clade's nodes end at it
    size = np.ones(tree_s.n_nodes, dtype=np.int64)
    for v in range(tree_s.n_nodes - 1):
        size[tree_s.parent[v]] += size[v]
    v = int(np.argmin(np.abs(size[:-1] - tips)))
    clade = np.arange(v - size[v] + 1, v + 1)
    rng = np.random.default_rng(2221)
    tree_s.length[:] = rng.exponential(1e3, size=tree_s.n_nodes)
    tree_s.length[clade] = rng.exponential(short, size=clade.size)
    tree_s.length[v] = 0.0
    # no long branch above the clade
    p = tree_s.parent[v]
    while p >= 0:
        tree_s.length[p] = 0.0
        p = tree_s.parent[p]
    tip_nodes = np.setdiff1d(np.arange(tree_s.n_nodes), tree_s.parent)
    inside = np.nonzero(np.isin(tip_nodes, clade))[0]
    counts = table_iid(64, tips, 0.1, seed=2222).dense()
    outside = np.setdiff1d(np.arange(tips), inside)
    counts[:32, outside] = 0.0
    counts[:32][counts[:32].sum(1) == 0, inside[0]] = 1.0
    check(tree_s, STable.from_dense(counts), f"clade of {short:g}")
