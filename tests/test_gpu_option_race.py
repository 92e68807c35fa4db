"""Options that another thread sets while calls run: a call goes by the values
it started with, so its result is one of those the settings give, bit for bit."""
import threading

import numpy as np
import pytest

import paper_2005_05826_gb300 as uf
from synth import table_iid, yule_tree

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("gpu_library")]

SETTINGS = [(48_000_000, 2), (200_000, 2), (48_000_000, 0), (200_000, 6)]


@pytest.mark.parametrize("method,precision", [("weighted_normalized", "mixed"), ("generalized", "mixed"),
                                              ("unweighted", "fp64")])
def test_region_size_and_fusing_change_while_calls_run(method, precision):
    tree_s = yule_tree(900, seed=2400)
    table_s = table_iid(640, 900, 0.01, seed=2401)
    tree = uf.Tree(tree_s.parent, tree_s.length)
    table = uf.Table(table_s.indptr, table_s.indices, table_s.data, tree)
    names = ("sparse_region_bytes", "sparse_fuse")

    def call():
        return np.asarray(uf.uf_compute(tree, table, method, 0.5, precision)[0])

    uf.uf_set_option("sparse", 2)
    stop = threading.Event()
    try:
        expected = []
        for values in SETTINGS:
            for name, v in zip(names, values):
                uf.uf_set_option(name, v)
            expected.append(call())
        # every branch is scattered, and integer sums do not depend on the order
        assert all((e == expected[0]).all() for e in expected)

        def toggle():
            k = 0
            while not stop.is_set():
                for name, v in zip(names, SETTINGS[k % len(SETTINGS)]):
                    uf.uf_set_option(name, v)
                k += 1

        t = threading.Thread(target=toggle)
        t.start()
        try:
            got = [call() for _ in range(150)]
        finally:
            stop.set()
            t.join()
        assert all((g == expected[0]).all() for g in got)
    finally:
        uf.uf_set_option("sparse", 1)
        uf.uf_set_option("sparse_region_bytes", 0)
        uf.uf_set_option("sparse_fuse", 2)
