"""Calls whose sample lists would not fit the device memory at hand scatter
without lists: the same table with the memory free and with all but a little of it
taken, both against the FP64 oracle.  In a process of its own, so that no earlier
call's pool memory counts as free."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]

CHILD = """
import sys
import numpy as np, torch
import oracle
import paper_2005_05826_gb300 as uf
from synth import pair_subset, table_iid, yule_tree
from tests.gpu_util import assert_close, condensed_index

method, precision, n, tips, density, left = sys.argv[1:]
n, tips, density, left = int(n), int(tips), float(density), int(left)


def handles(n, tips, density):
    tree_s = yule_tree(tips, seed=2500)
    table_s = table_iid(n, tips, density, seed=2501)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    return tree_s, table_s, tree, uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)


out = torch.empty(n * (n - 1) // 2, dtype=torch.float64, device="cuda")
uf.uf_set_option("sparse", 2)
tree_s, table_s, tree, table = handles(n, tips, density)
i, j = pair_subset(n, 4000, seed=12345)
exp = oracle.pairs(tree_s, table_s, method, 0.5, i, j)[0]
idx = condensed_index(n, i, j)
# every kernel loaded before the memory goes: lists, tiles and the direct scatter
small = handles(600, 400, 0.02)
for sparse in (2, 1, 0):
    uf.uf_set_option("sparse", sparse)
    uf.uf_compute(*small[2:], method, 0.5, precision)
    uf.uf_compute_ranges(small[2], [(small[3], 0, 300), (small[3], 0, 1)], method, 0.5, precision)
# (the handles' device copies are made at their first use: here, without lists and in small blocks)
uf.uf_set_option("branch_block", 256)
uf.uf_compute(tree, table, method, 0.5, precision, 0, 1)
uf.uf_set_option("branch_block", 0)
uf.uf_set_option("sparse", 2)
torch.cuda.synchronize()
hold = []
free = torch.cuda.mem_get_info()[0]
hold.append(torch.empty(free - left * (1 << 20), dtype=torch.uint8, device="cuda"))
_, rep_short = uf.uf_compute(tree, table, method, 0.5, precision, out=out)
assert_close(out.cpu().numpy()[idx], exp, method, precision, f"{left} MiB left")
hold.clear()
torch.cuda.empty_cache()
out.fill_(-1.0)
_, rep = uf.uf_compute(tree, table, method, 0.5, precision, out=out)
assert_close(out.cpu().numpy()[idx], exp, method, precision, "memory free")
print("sparse rows", rep_short.sparse_rows, "with little memory,", rep.sparse_rows, "with more")
# without lists a branch of more than 4,096 entries is dense
assert 0 < rep_short.sparse_rows < rep.sparse_rows
"""


@pytest.mark.parametrize("method,precision,n,tips,density,left",
                         [("weighted_normalized", "mixed", 2048, 20_000, 0.03, 200),
                          ("generalized", "mixed", 1024, 20_000, 0.05, 200),
                          ("weighted_normalized", "fp64", 1300, 20_000, 0.04, 300)])
def test_lists_larger_than_the_memory_at_hand(method, precision, n, tips, density, left):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, method, precision, str(n), str(tips), str(density), str(left)],
                       cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
