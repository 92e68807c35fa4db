"""The calls whose speed counts: UniFrac matrices as a user of this package computes them.

A case says which entry point is called, on a tree and a table of which shape, with which
method and precision.  Trees are Yule trees with Exp(mean 0.1) branch lengths; tables hold
integer counts, 1 + Poisson(LogNormal(1, 1)) or, heavy-tailed, max(1, round(LogNormal(1, 1.5))),
at a feature prevalence that is the same for every feature ("density") or Beta-distributed, the
shapes of this repository's workloads.

Keys of a case:
  call        "compute" (uf_compute into a CUDA tensor), "ranges" (uf_compute_ranges: one matrix
              per table of a batch), "batch" (uf_compute_batch), "noalloc" (uf_compute_noalloc),
              "script" (host arrays in, handles made, host matrix out)
  n, tips     samples and tree tips ("ranges" and "batch": `tables` tables of lo .. hi samples)
  beta_a, beta_b / density, heavy    the table's prevalence and counts
  method, alpha, precision           as the entry points take them; mixed calls give FP32 results
  start, stop                        stripe range (0, 0: the whole condensed matrix)
  stream                             on a stream of its own (the call returns once it is enqueued)
                                     or on the default one
"""
import contextlib
import math

import numpy as np
import torch

import paper_2005_05826_gb300 as uf

_SHAPE = dict(beta_a=0.0, beta_b=0.0, density=0.0, heavy=False)
_CALL = dict(alpha=1.0, start=0, stop=0, stream=False)


def _case(name, call, n, tips, method, precision, **more):
    return {"name": name, "call": call, "n": n, "tips": tips, "method": method, "precision": precision,
            **_SHAPE, **_CALL, **more}


def listed():
    study = dict(beta_a=0.5, beta_b=20.0)
    return [
        # a first look at a small study: the smallest table this repository is tested on, in the
        # binding's default precision; latency is all that counts
        _case("tiny_unweighted_fp64", "compute", 64, 1024, "unweighted", "fp64", density=0.1),
        # a service that may not enter the device allocator
        _case("noalloc_weighted_fp64", "noalloc", 61, 1000, "weighted_normalized", "fp64", density=0.1),
        # an analysis script: arrays from a file, one call with the defaults, a numpy matrix
        _case("script_weighted_fp64", "script", 301, 12_000, "weighted_normalized", "fp64", density=0.02),
        # an ordinary study (2,048 samples, 50,000 tips), method by method
        _case("study_unweighted_mixed", "compute", 2048, 50_000, "unweighted", "mixed", stream=True, **study),
        _case("study_weighted_mixed", "compute", 2048, 50_000, "weighted_normalized", "mixed", stream=True, **study),
        _case("study_generalized_mixed", "compute", 1003, 50_000, "generalized", "mixed", alpha=0.5, stream=True,
              **study),
        # the same kind of study where the FP64 result is wanted (the default)
        _case("study_unweighted_fp64", "compute", 2048, 50_000, "unweighted", "fp64", **study),
        _case("study_weighted_fp64", "compute", 1531, 50_000, "weighted_unnormalized", "fp64", **study),
        _case("study_generalized_fp64", "compute", 500, 20_000, "generalized", "fp64", alpha=0.5, **study),
        # many tables over one tree in one call (rarefactions, body sites)
        _case("batch_weighted_mixed", "ranges", 0, 100_000, "weighted_normalized", "mixed", density=0.01, tables=8,
              lo=203, hi=1000, stream=True),
        # a whole large study: 25,000 samples, 300,000 tips, every pair
        _case("large_unweighted_mixed", "compute", 25_000, 300_000, "unweighted", "mixed", beta_a=0.1, beta_b=19.9,
              heavy=True, stream=True),
        # one job of the largest: 113,000 samples, 500,000 tips, a stripe range of the matrix
        _case("largest_range_weighted_mixed", "compute", 113_000, 500_000, "weighted_normalized", "mixed",
              beta_a=0.06, beta_b=19.94, heavy=True, stop=2048, stream=True),
    ]


_METHODS = ("unweighted", "weighted_normalized", "weighted_unnormalized", "generalized", "unweighted_unnormalized",
            "vaw_weighted_normalized", "vaw_weighted_unnormalized")


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["compute"] * 5 + ["ranges", "batch", "noalloc", "script", "wide"])
    method = rng.choice(_METHODS[:4] * 2 + _METHODS[4:])
    precision = rng.choice(["mixed", "fp64"])
    n, tips, stop = _log_int(rng, 2, 2048), _log_int(rng, 60, 50_000), 0
    more = {"stream": rng.random() < 0.6}
    if method == "generalized":
        more["alpha"] = rng.choice([0.5, 0.5, 0.25, 0.0])
    if rng.random() < 0.6:
        b = rng.uniform(10.0, 25.0)
        more.update(beta_a=b * math.exp(rng.uniform(math.log(0.004), math.log(0.03))), beta_b=b)
    else:
        more["density"] = math.exp(rng.uniform(math.log(0.004), math.log(0.1)))
    more["heavy"] = rng.random() < 0.3
    if call == "wide":  # a stripe range of a large table
        call, method, precision = "compute", rng.choice(_METHODS[:3]), "mixed"
        n, tips = _log_int(rng, 4000, 20_000), _log_int(rng, 20_000, 200_000)
        stop = rng.randint(200, 2000)
        more.pop("alpha", None)
        more.update(start=rng.randint(0, 150), density=0.0, beta_a=0.1, beta_b=19.9, heavy=True)
    elif call == "noalloc":  # everything fits 64 MiB
        n, tips, precision, method = _log_int(rng, 4, 100), _log_int(rng, 60, 3000), "fp64", rng.choice(_METHODS[:4])
        more["alpha"] = 0.5 if method == "generalized" else 1.0
    elif call == "script":
        n, tips = _log_int(rng, 10, 600), _log_int(rng, 200, 20_000)
    elif call in ("ranges", "batch"):
        if call == "batch":
            precision = "fp64"
        more.update(tables=rng.randint(2, 9), lo=_log_int(rng, 20, 150), hi=_log_int(rng, 160, 800))
        n, tips = 0, _log_int(rng, 2000, 50_000)
    if precision == "fp64" and (method == "generalized" or method.startswith("vaw")):
        # the costliest combinations: no larger than the largest listed ones
        n, tips = min(n, 500), min(tips, 20_000)
        if call in ("ranges", "batch"):
            more.update(tables=min(more["tables"], 4), hi=min(more["hi"], 300))
    c = _case("", call, n, tips, method, precision, **{**more, "stop": stop})
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _tree(tips, rng):
    """A Yule tree in postorder: a clade of m tips splits into i and m - i, i uniform on 1 .. m - 1."""
    parent = np.full(2 * tips - 1, -1, dtype=np.int64)
    at, m, up = np.zeros(1, np.int64), np.full(1, tips, np.int64), np.full(1, -1, np.int64)
    while at.size:
        node = at + 2 * m - 2
        parent[node] = up
        at, m, node = at[m > 1], m[m > 1], node[m > 1]
        left = 1 + np.floor(rng.random(m.size) * (m - 1)).astype(np.int64)
        at, m, up = (np.concatenate([at, at + 2 * left - 1]), np.concatenate([left, m - left]),
                     np.concatenate([node, node]))
    return parent, rng.exponential(0.1, size=parent.size)


def _table(n, case, rng):
    """CSR counts (host arrays), drawn on the GPU."""
    dev, tips = torch.device("cuda"), case["tips"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(rng.integers(1 << 62)))
    prev = np.full(tips, case["density"]) if case["density"] else rng.beta(case["beta_a"], case["beta_b"], size=tips)
    per = torch.from_numpy(rng.binomial(n, prev)).to(dev)
    feature = torch.repeat_interleave(torch.arange(tips, device=dev), per)
    sample = torch.randint(0, n, (feature.numel(),), device=dev, generator=gen)
    empty = torch.nonzero(torch.bincount(sample, minlength=n) == 0).reshape(-1)  # these get one feature
    more = torch.randint(0, tips, (empty.numel(),), device=dev, generator=gen)
    key = torch.unique(torch.cat([sample * tips + feature, empty * tips + more]))
    sample, feature = key // tips, (key % tips).to(torch.int32)
    z = torch.randn(key.numel(), dtype=torch.float64, device=dev, generator=gen)
    if case["heavy"]:
        counts = torch.clamp(torch.round(torch.exp(1.0 + 1.5 * z)), min=1.0)
    else:
        counts = 1.0 + torch.poisson(torch.exp(1.0 + z), generator=gen)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    indptr[1:] = torch.cumsum(torch.bincount(sample, minlength=n), 0)
    return indptr.cpu().numpy(), feature.cpu().numpy(), counts.cpu().numpy()


def _sizes(case):
    if not case["n"]:
        return [int(x) for x in np.geomspace(case["lo"], case["hi"], case["tables"])]
    return [case["n"]]


def _inputs(case, seed):
    rng = np.random.default_rng([seed, 2005])
    return _tree(case["tips"], rng), [_table(n, case, rng) for n in _sizes(case)]


def _range(case, n):
    return (case["start"], case["stop"]) if case["stop"] else (0, n // 2)


def _values(case, n):
    s0, s1 = _range(case, n)
    return n * (n - 1) // 2 if (s0, s1) == (0, n // 2) else (s1 - s0) * n


def prepare(case, seed):
    (parent, length), tables = _inputs(case, seed)
    if case["call"] == "script":
        return {"case": case, "parent": parent, "length": length, "table": tables[0]}
    tree = uf.Tree(parent, length)
    dtype = torch.float32 if case["precision"] == "mixed" and case["call"] != "batch" else torch.float64
    return {"case": case, "tree": tree, "tables": [uf.Table(*t, tree) for t in tables],
            "outs": [torch.empty(_values(case, n), dtype=dtype, device="cuda") for n in _sizes(case)],
            "stream": torch.cuda.Stream() if case["stream"] else None}


def run(state):
    c = state["case"]
    method, alpha, precision = c["method"], c["alpha"], c["precision"]
    if c["call"] == "script":
        tree = uf.Tree(state["parent"], state["length"])
        table = uf.Table(*state["table"], tree)
        return uf.uf_compute(tree, table, method, alpha, precision, out_fp32=precision == "mixed")[0]
    tree, tables, outs = state["tree"], state["tables"], state["outs"]
    fp32 = outs[0].dtype == torch.float32
    with torch.cuda.stream(state["stream"]) if state["stream"] is not None else contextlib.nullcontext():
        if c["call"] == "noalloc":
            return uf.uf_compute_noalloc(tree, tables[0], method, alpha, precision, out=outs[0])
        if c["call"] == "batch":
            return uf.uf_compute_batch(tree, tables, method, alpha, precision, outs=outs)[0]
        if c["call"] == "ranges":
            jobs = [(t, *_range(c, t.n_samples)) for t in tables]
            return uf.uf_compute_ranges(tree, jobs, method, alpha, precision, outs=outs, out_fp32=fp32)[0]
        start, stop = _range(c, c["n"])
        return uf.uf_compute(tree, tables[0], method, alpha, precision, start, stop, out=outs[0], out_fp32=fp32)[0]


def work(case):
    """Bytes: the table's entries (sample, feature and count: 12), the branch lengths, the results.  Flops: per pair
    and branch of the tree that joins the tips either sample has (at least 2 m - 1 branches for m tips), the term and
    its sum."""
    tips = case["tips"]
    prev = case["density"] or case["beta_a"] / (case["beta_a"] + case["beta_b"])
    size = 4 if case["precision"] == "mixed" and case["call"] != "batch" else 8
    nbytes, flops = 8.0 * (2 * tips - 1), 0.0
    for n in _sizes(case):
        per_sample = max(1.0, tips * prev)
        nbytes += 12.0 * n * per_sample + float(size) * _values(case, n)
        flops += 2.0 * _values(case, n) * (2.0 * per_sample - 1.0)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the definition in 64 bits

def _tip_ranges(parent):
    """Tips [lo, hi) below every node (postorder: a clade's nodes end at its own)."""
    n = parent.size
    has_child = np.zeros(n, dtype=bool)
    has_child[parent[:-1]] = True
    hi = np.cumsum(~has_child)
    size = np.ones(n, dtype=np.int64)  # nodes of the clade; a clade of m tips has 2 m - 1
    for v in range(n - 1):
        p = parent[v]
        size[p] += size[v]
    return hi - (size + 1) // 2, hi


def _terms(method, alpha, p_i, p_j, c_i, c_j, t_i, t_j, length):
    """(numerator, denominator) over the branches of the last axis, [rows, samples]."""
    if method == "generalized":
        s, d = p_i + p_j, (p_i - p_j).abs_()
        if alpha == 0.5:
            root = s.sqrt_()
            d = torch.where(root > 0, d / root, d)
            return d @ length, root @ length
        w = torch.where(s > 0, s.pow(alpha - 1.0), torch.zeros_like(s))
        return (d * w) @ length, (s * w) @ length
    below, rest = c_i + c_j, (t_i - c_i) + (t_j - c_j)
    w = below.mul_(rest)
    w = torch.where(w > 0, w.rsqrt(), torch.zeros_like(w))
    return ((p_i - p_j).abs() * w) @ length, ((p_i + p_j) * w) @ length


def _matrix(case, parent, length, table):
    """The n x n distances of one table, from the definition."""
    dev, method = torch.device("cuda"), case["method"]
    indptr, indices, data = (torch.from_numpy(x).to(dev) for x in table)
    n, tips = indptr.numel() - 1, case["tips"]
    lo, hi = (torch.from_numpy(x).to(dev) for x in _tip_ranges(parent))
    length = torch.from_numpy(length).to(dev)
    counts = torch.zeros((n, tips + 1), dtype=torch.float64, device=dev)
    rows = torch.repeat_interleave(torch.arange(n, device=dev), indptr[1:] - indptr[:-1])
    counts[rows, indices.long() + 1] = data
    total = counts.sum(1, keepdim=True)
    below = torch.cumsum(counts, 1)  # whole numbers: sums below a node are exact differences
    num = torch.zeros((n, n), dtype=torch.float64, device=dev)
    den = torch.zeros_like(num)
    wide = method.startswith("vaw") or method == "generalized"
    step = max(64, min(4096, (1 << 26) // max(1, n))) if wide else 4096
    for v in range(0, parent.size - 1, step):
        w = min(parent.size - 1, v + step)
        c, l = below[:, hi[v:w]] - below[:, lo[v:w]], length[v:w]
        p = c / total
        if wide:
            r = max(1, (1 << 26) // (n * (w - v)))
            for i in range(0, n, r):
                a, b = _terms(method, case["alpha"], p[i:i + r, None], p[None], c[i:i + r, None], c[None],
                              total[i:i + r, None], total[None], l)
                num[i:i + r] += a
                den[i:i + r] += b
        elif method.startswith("unweighted"):
            a = (c > 0).double()
            both, own = (a * l) @ a.T, a @ l
            num += (a * l) @ (1 - a).T + ((1 - a) * l) @ a.T
            den += own[:, None] + own[None] - both
        else:
            num += torch.cdist(p * l, p * l, p=1.0)
            own = p @ l
            den += own[:, None] + own[None]
    if method.endswith("unnormalized"):
        return num
    return torch.where(den > 0, num / den, torch.zeros_like(num))


def exact(case, seed):
    cells = sum(n * n for n in _sizes(case)) * (2.0 * case["tips"] - 1)
    each = 1.0
    if case["method"].startswith("vaw") or case["method"] == "generalized":
        each = 4.0 if case["alpha"] in (0.5, 1.0) else 12.0
    if cells * each > 6e11:
        return None
    (parent, length), tables = _inputs(case, seed)
    found = []
    for table in tables:
        n = table[0].size - 1
        d = _matrix(case, parent, length, table)
        if _range(case, n) == (0, n // 2):
            i, j = torch.triu_indices(n, n, 1, device=d.device)
        else:
            s = torch.arange(*_range(case, n), device=d.device)[:, None]
            i = torch.arange(n, device=d.device)[None].expand(s.numel(), n)
            j = (i + s + 1) % n
        found.append(d[i, j].reshape(-1).cpu())
    return found if case["call"] in ("ranges", "batch") else found[0]
