"""Cases that a user of the biased graph-attention library runs, through its public entry points.

A case names one call, or the few calls that belong together, on a packed batch of graphs:

  step     gt_spd_build, gt_biased_attn_fwd and gt_biased_attn_bwd: one training step on a batch
  spd      gt_spd_build: the structural encoding of a new batch, from its CSR
  fwd      gt_biased_attn_fwd (inference, and the first half of training)
  bwd      gt_biased_attn_bwd
  chunked  gt_biased_attn_fwd_chunked: the forward one key/value chunk at a time
  codes    categorical pair features: gt_feature_encode, then forward and backward through the code matrix
  feature  arbitrary pair features: gt_feature_attn_fwd and gt_feature_attn_bwd

Fields: `graph` (er Erdos-Renyi, ba preferential attachment, pl power law, rgg random geometric, directed: a directed
Erdos-Renyi graph) with average degree `degree`; `graphs` graphs of `n_min` to `n_max` nodes, whose sizes follow from
`sizes`, so that the work does not depend on the seed; `heads`, `head_dim`, `max_dist`; `chunks` key/value chunks;
`vectors` distinct feature vectors.
"""
import math
import random

import numpy as np
import torch

from paper_2609_34420_b200 import binding as gt
from paper_2609_34420_b200 import workloads as wl


def _case(what, graph, degree, n_min, n_max, heads, head_dim, max_dist, graphs=1, sizes=0, chunks=1, vectors=0):
    return {"what": what, "graph": graph, "degree": degree, "graphs": graphs, "n_min": n_min, "n_max": n_max, "sizes": sizes,
            "heads": heads, "head_dim": head_dim, "max_dist": max_dist, "chunks": chunks, "vectors": vectors}


def listed():
    cases = {
        # The smallest training step: one sampled sub-graph of 256 nodes with few, narrow heads.  Launches and host
        # work count here, not rates.
        "step_er256": _case("step", "er", 8, 256, 256, 4, 32, 8),
        # The encoding of one ordinary batch: a sampled sub-graph with hubs, four levels deep.
        "spd_ba4096": _case("spd", "ba", 10, 4096, 4096, 8, 64, 16),
        # The encoding of many small graphs of large diameter (meshes, molecules, road maps) in one packed batch; every
        # graph has another size, so pitches and row tails are ragged.
        "spd_rgg64": _case("spd", "rgg", 6, 512, 2048, 16, 64, 12, graphs=64),
        # The encoding of a whole citation graph at once: the largest matrix, 4 GiB.
        "spd_pl65536": _case("spd", "pl", 12, 65536, 65536, 8, 64, 24),
        # Forward and backward of an ordinary batch.
        "fwd_ba4096": _case("fwd", "ba", 10, 4096, 4096, 8, 64, 16),
        "bwd_ba4096": _case("bwd", "ba", 10, 4096, 4096, 8, 64, 16),
        # Forward and backward of the packed batch of small ragged graphs.
        "fwd_rgg64": _case("fwd", "rgg", 6, 512, 2048, 16, 64, 12, graphs=64),
        "bwd_rgg64": _case("bwd", "rgg", 6, 512, 2048, 16, 64, 12, graphs=64),
        # The whole graph: the forward as context parallelism sees it, in eight key/value chunks, and the backward.
        "chunked_pl65536": _case("chunked", "pl", 12, 65536, 65536, 8, 64, 24, chunks=8),
        "bwd_pl65536": _case("bwd", "pl", 12, 65536, 65536, 8, 64, 24),
        # A training step with categorical pair features (edge type, hop class and the like) on the largest sampled
        # batch: encoding, forward with the fp32 output, backward, gradient of the feature weights.
        "codes_8192": _case("codes", "", 0, 8192, 8192, 8, 64, 0, vectors=12),
        # Forward and backward with pair features that take any values, on a small sampled batch.
        "feature_1500": _case("feature", "", 0, 1500, 1500, 8, 64, 0),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _spread(rng, lo, hi):
    """A whole number from lo to hi, even over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _packed(rng, what, graph, degree, max_graphs, n_lo, n_hi):
    """A packed batch of at most about 90 000 nodes in graphs of n_lo to n_hi nodes."""
    n_max = _spread(rng, 2 * n_lo, n_hi)
    n_min = _spread(rng, n_lo, n_max)
    graphs = min(_spread(rng, 2, max_graphs), max(2, 90000 // n_max))
    return _case(what, graph, degree, n_min, n_max, rng.choice((2, 4, 8, 16)), rng.choice((32, 64, 64)),
                 rng.randint(4, 24), graphs=graphs, sizes=rng.randrange(1 << 20))


def draw(rng):
    what = rng.choice(("step", "spd", "spd", "fwd", "bwd", "chunked", "codes", "feature"))
    if what == "step":
        if rng.random() < 0.5:
            return _packed(rng, what, "er", rng.randint(3, 8), 64, 16, 300)
        n = _spread(rng, 64, 2048)
        return _case(what, "er", rng.randint(3, 12), n, n, rng.choice((2, 4, 8)), rng.choice((32, 64)), rng.randint(4, 20))
    if what == "codes":
        n = _spread(rng, 1000, 8192)
        return _case(what, "", 0, n, n, rng.choice((4, 8)), rng.choice((32, 64)), 0, vectors=_spread(rng, 4, 200))
    if what == "feature":
        n = _spread(rng, 500, 4096)
        return _case(what, "", 0, n, n, rng.choice((4, 8)), rng.choice((32, 64)), 0)
    if what == "chunked":
        n = _spread(rng, 4096, 65536)
        return _case(what, "pl", rng.randint(8, 14), n, n, rng.choice((4, 8)), rng.choice((32, 64, 64)), rng.randint(8, 24),
                     chunks=rng.randint(2, 8))
    if rng.random() < 0.4:
        return _packed(rng, what, "rgg", rng.randint(4, 8), 64, 128, 4096)
    n = _spread(rng, 1000, 65536)
    graph = "pl" if n > 8192 else rng.choice(("ba", "pl", "directed"))
    # Large power-law graphs are shallow: more than 24 levels are asked for on smaller graphs only.
    return _case(what, graph, 2 * rng.randint(3, 7), n, n, rng.choice((4, 8)), rng.choice((32, 64, 64)),
                 rng.randint(4, 24 if n > 16384 else 40))


def _sizes(case):
    if case["graphs"] == 1:
        return [case["n_max"]]
    rng = np.random.Generator(np.random.PCG64(case["sizes"]))
    return [int(n) for n in rng.integers(case["n_min"], case["n_max"] + 1, size=case["graphs"])]


def _graph(case, n, seed):
    kind, degree = case["graph"], case["degree"]
    if kind == "er":
        return wl.erdos_renyi(n, min(1.0, degree / max(n - 1, 1)), seed)
    if kind == "ba":
        return wl.barabasi_albert(n, degree // 2, seed)
    if kind == "pl":
        return wl.chung_lu_power_law(n, float(degree), 2.1, seed)
    if kind == "rgg":
        return wl.random_geometric(n, float(degree), seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    return wl.csr_from_edges(n, rng.integers(0, n, size=n * degree), rng.integers(0, n, size=n * degree), symmetric=False)


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    rng = torch.Generator(device=dev).manual_seed(seed)
    what, H, d, D = case["what"], case["heads"], case["head_dim"], case["max_dist"]
    sizes = _sizes(case)
    T = sum(sizes)
    s = {"case": case}

    def normal(std=1.0):
        return (torch.randn(T, H, d, device=dev, generator=rng) * std).bfloat16()

    def like(*shape, dtype=torch.float32):
        return torch.empty(*shape, dtype=dtype, device=dev)

    if what != "spd":
        s["q"], s["k"], s["v"], s["do"] = normal(), normal(), normal(), normal()
        s["out"], s["lse"] = torch.empty_like(s["q"]), like(H, T)
        s["dq"], s["dk"], s["dv"] = (torch.empty_like(s["q"]) for _ in range(3))

    if what in ("codes", "feature"):
        s["batch"] = batch = gt.Batch(T)
        s["weights"] = torch.randn(H, 4, device=dev, generator=rng) * 0.01
        s["dweights"] = torch.empty_like(s["weights"])
        if what == "feature":
            s["features"] = torch.randint(0, 256, (T, T, 4), device=dev, generator=rng, dtype=torch.uint8)
            s["ws_bwd"] = gt._workspace(gt.gt_feature_attn_bwd_workspace(batch, H), dev)
            return s
        # Distinct vectors, as a categorical encoding has them: the first feature numbers them, the others are arbitrary.
        vec = torch.randint(0, 256, (case["vectors"], 4), device=dev, generator=rng, dtype=torch.uint8)
        vec[:, 0] = torch.arange(case["vectors"], device=dev, dtype=torch.uint8)
        pick = torch.randint(0, case["vectors"], (T, T), device=dev, generator=rng)
        s["features"] = vec[pick]
        width = max(case["vectors"], 3)
        s["codes"] = like(T * wl.round_up(T, 16), dtype=torch.uint8)
        s["vectors"] = like(256, dtype=torch.int32)
        s["table"], s["dtable"] = like(H, width), like(H, width)
        s["out32"] = like(T, H, d)
        s["ws_enc"] = gt._workspace(gt.lib().gt_feature_encode_workspace(), dev)
        s["ws_fwd"] = gt._workspace(gt.gt_biased_attn_fwd_workspace(batch, H, d), dev)
        s["ws_bwd"] = gt._workspace(gt.gt_biased_attn_bwd_workspace(batch, H, d, width - 2), dev)
        return s

    g = wl.pack_graphs([_graph(case, n, seed * 4099 + i) for i, n in enumerate(sizes)])
    single = g.n_graphs == 1
    s["batch"] = batch = gt.Batch(T, g.n_graphs, g.max_seqlen,
                                  None if single else torch.from_numpy(g.cu_seqlens).to(dev),
                                  None if single else torch.from_numpy(g.spd_offsets).to(dev))
    s["row_ptr"], s["col_idx"] = torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col_idx).to(dev)
    s["spd"] = like(g.spd_bytes, dtype=torch.uint8)
    s["ws_spd"] = gt._workspace(gt.gt_spd_build_workspace(batch, len(g.col_idx), D), dev)
    if what == "spd":
        return s
    s["bias"] = torch.randn(H, D + 2, device=dev, generator=rng) * 0.5
    s["dbias"] = torch.empty_like(s["bias"])
    s["ws_fwd"] = gt._workspace(gt.gt_biased_attn_fwd_workspace(batch, H, d), dev)
    if what == "chunked":
        s["ws_chunked"] = gt._workspace(gt.gt_biased_attn_fwd_chunked_workspace(batch, H, d, case["chunks"]), dev)
    if what in ("step", "bwd"):
        s["ws_bwd"] = gt._workspace(gt.gt_biased_attn_bwd_workspace(batch, H, d, D), dev)
    if what != "step":
        gt.gt_spd_build(s["row_ptr"], s["col_idx"], batch, D, s["spd"], s.pop("ws_spd"))
    if what == "bwd":
        gt.gt_biased_attn_fwd(s["q"], s["k"], s["v"], s["spd"], s["bias"], batch, D, s["out"], s["lse"], s["ws_fwd"])
    return s


def run(s):
    case, batch = s["case"], s["batch"]
    what, D = case["what"], case["max_dist"]
    if what == "feature":
        gt.gt_feature_attn_fwd(s["q"], s["k"], s["v"], s["features"], s["weights"], batch, s["out"], s["lse"])
        gt.gt_feature_attn_bwd(s["q"], s["k"], s["v"], s["do"], s["lse"], s["features"], s["weights"], batch,
                               s["dq"], s["dk"], s["dv"], s["dweights"], s["ws_bwd"])
        return [s[x] for x in ("out", "lse", "dq", "dk", "dv", "dweights")]
    if what == "codes":
        width = s["table"].shape[1]
        gt.gt_feature_encode(s["features"], batch, s["codes"], s["vectors"], s["ws_enc"])
        gt.gt_feature_code_table(s["weights"], s["vectors"], s["table"])
        gt.gt_biased_attn_fwd_ex(s["q"], s["k"], s["v"], s["codes"], s["table"], batch, width - 2, s["out"], s["lse"],
                                 s["out32"], s["ws_fwd"])
        gt.gt_biased_attn_bwd_ex(s["q"], s["k"], s["v"], s["out"], s["do"], s["lse"], s["codes"], s["table"], batch,
                                 width - 2, s["dq"], s["dk"], s["dv"], s["dtable"], s["out32"], s["ws_bwd"])
        gt.gt_feature_code_dweights(s["dtable"], s["vectors"], s["dweights"])
        return [s[x] for x in ("codes", "vectors", "out", "out32", "lse", "dq", "dk", "dv", "dtable", "dweights")]
    if what in ("step", "spd"):
        gt.gt_spd_build(s["row_ptr"], s["col_idx"], batch, D, s["spd"], s["ws_spd"])
        if what == "spd":
            return s["spd"]
    if what in ("step", "fwd"):
        gt.gt_biased_attn_fwd(s["q"], s["k"], s["v"], s["spd"], s["bias"], batch, D, s["out"], s["lse"], s["ws_fwd"])
        if what == "fwd":
            return s["out"], s["lse"]
    if what == "chunked":
        gt.gt_biased_attn_fwd_chunked(s["q"], s["k"], s["v"], s["spd"], s["bias"], batch, D, s["out"], s["lse"],
                                      case["chunks"], None, s["ws_chunked"])
        return s["out"], s["lse"]
    gt.gt_biased_attn_bwd(s["q"], s["k"], s["v"], s["out"], s["do"], s["lse"], s["spd"], s["bias"], batch, D,
                          s["dq"], s["dk"], s["dv"], s["dbias"], s["ws_bwd"])
    grads = [s[x] for x in ("dq", "dk", "dv", "dbias")]
    return [s["spd"], s["out"], s["lse"]] + grads if what == "step" else grads


def work(case):
    """Two contractions forward and five backward over the pairs of each graph; every tensor once, a pair's byte (or
    its four features) once for each pass that uses it."""
    what, H, d = case["what"], case["heads"], case["head_dim"]
    sizes = _sizes(case)
    T, pairs = sum(sizes), sum(n * n for n in sizes)
    matrix = sum(n * wl.round_up(n, 16) for n in sizes)
    csr = 4 * (T + 1) + 4 * T * case["degree"]
    tensor, rows = 2 * T * H * d, 4 * T * H
    fwd = {"bytes": 4 * tensor + rows, "flops": 4 * H * d * pairs}
    bwd = {"bytes": 8 * tensor + rows, "flops": 10 * H * d * pairs}
    if what == "spd":
        return {"bytes": matrix + csr, "flops": 0}
    if what in ("fwd", "chunked"):
        return {"bytes": fwd["bytes"] + matrix, "flops": fwd["flops"]}
    if what == "bwd":
        return {"bytes": bwd["bytes"] + matrix, "flops": bwd["flops"]}
    both = {"bytes": fwd["bytes"] + bwd["bytes"], "flops": fwd["flops"] + bwd["flops"]}
    if what == "step":
        return {"bytes": both["bytes"] + 3 * matrix + csr, "flops": both["flops"]}
    if what == "codes":
        return {"bytes": both["bytes"] + 4 * pairs + 3 * matrix + 8 * T * H * d, "flops": both["flops"]}
    return {"bytes": both["bytes"] + 8 * pairs, "flops": both["flops"]}


def tolerance(case):
    # Distances are whole numbers.  Attention multiplies bf16 operands (probabilities and score gradients among them) and
    # rounds its results to bf16.
    return "exact" if case["what"] == "spd" else {"rel": 1e-2}
