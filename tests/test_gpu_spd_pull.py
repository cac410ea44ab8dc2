"""Where the pull forms of gt_spd_build change their course: bit-exact against the BFS oracle."""
import numpy as np
import pytest

from paper_2609_34420_b200 import workloads as wl

from test_gpu_spd import check, pytestmark  # noqa: F401  (GPU tests)


def directed(n, m, seed, hub_edges=0, hubs=1):
    """Random directed graph with isolated vertices at the end and a few vertices of many out-edges."""
    rng = np.random.Generator(np.random.PCG64(seed))
    src, dst = rng.integers(0, n - n // 20, m), rng.integers(0, n - n // 25, m)
    for h in range(hubs if hub_edges else 0):
        src = np.concatenate([src, np.full(hub_edges, 3 * h)])
        dst = np.concatenate([dst, rng.choice(n - n // 30, hub_edges, replace=False)])
    return wl.csr_from_edges(n, src, dst, symmetric=False)


def one(csr, D):
    check(wl.Workload("one", wl.pack_graphs([csr]), 1, 32, D))


@pytest.mark.parametrize("D", [1, 2, 7, 15, 254])        # code planes: 2, 2, 4, 5, 8
def test_a_batch_of_wide_rows(D):
    """Enough targets for blocks of 128 (64 with eight planes): ragged sizes, deep undirected graphs, a path, isolated nodes."""
    rng = np.random.Generator(np.random.PCG64(D))
    graphs = [wl.random_geometric(int(n), 5.0, 100 + i) for i, n in enumerate(rng.integers(900, 1100, 40))]
    path = np.arange(699)
    graphs[7] = wl.csr_from_edges(700, path, path + 1, symmetric=False)
    graphs[9] = (np.zeros(34, np.int32), np.zeros(0, np.int32))
    check(wl.Workload("wide", wl.pack_graphs(graphs), 1, 32, D))


def test_more_graphs_than_are_sorted_by_size():
    rng = np.random.Generator(np.random.PCG64(5))
    check(wl.small_workload([int(n) for n in rng.integers(1, 70, 300)], 1, 32, 5, seed=2, avg_degree=2.0, directed=True))


def test_a_graph_whose_edges_do_not_fit_beside_sparse_ones():
    """The batch's average degree promises room for the largest graph's list; this one has 40 times as many edges, and hubs."""
    graphs = [wl.random_geometric(1000, 4.0, i) for i in range(30)] + [directed(1400, 90000, 3, hub_edges=900, hubs=3)]
    check(wl.Workload("outlier", wl.pack_graphs(graphs), 1, 32, 6))


@pytest.mark.parametrize("n,m,D", [(5600, 80000, 1), (6001, 90000, 5), (7000, 9000, 30), (14100, 60000, 20), (14128, 60000, 20), (14200, 60000, 20),
                                   (18941, 50000, 9)])
def test_one_graph_with_lists_in_the_workspace(n, m, D):
    """Hubs beyond a group's degree (some more than are kept in shared memory), sparse directed graphs of many levels,
    the last target block ragged, two blocks per SM (up to 14 126 nodes) and one."""
    one(directed(n, m, n, hub_edges=300, hubs=450 if n == 6001 else 2), D)


@pytest.mark.parametrize("n,degree", [(5600, 128), (14500, 33)])
def test_one_graph_with_too_many_edges_for_lists_in_the_workspace(n, degree):
    """More than 126 edges per vertex: the push; more than 32 from 14 500 nodes on: the bit matrices."""
    one(directed(n, n * degree, n), 3)


def test_one_deep_undirected_graph_with_lists_in_the_workspace():
    one(wl.random_geometric(9000, 6.5, 4), 9)


@pytest.mark.parametrize("n,m,D", [(18945, 46000, 11), (19200, 24000, 254), (19457, 400000, 2)])
def test_one_graph_beyond_the_pull(n, m, D):
    """The bit matrices at their smallest: more levels than level bits, a clip above them, rows that close early, isolated nodes."""
    one(directed(n, m, n, hub_edges=5000, hubs=2), D)


def shuffled(csr, seed):
    rp, ci = csr
    n = len(rp) - 1
    to = np.random.Generator(np.random.PCG64(seed)).permutation(n)
    return wl.csr_from_edges(n, to[np.repeat(np.arange(n), np.diff(rp))], to[ci], symmetric=False)


def long_ways(n, kind, seed):
    """Graphs hundreds to thousands of edges across."""
    i = np.arange(n)
    if kind == "ring":
        return wl.csr_from_edges(n, i, (i + 1) % n, symmetric=True)
    if kind == "directed ring":
        return shuffled(wl.csr_from_edges(n, i, (i + 1) % n, symmetric=False), seed)
    if kind == "one way":                    # a path with some of its reverse edges missing: components of edges both ways, in a row
        both = wl.csr_from_edges(n, np.concatenate([i[:-1], i[1:]]), np.concatenate([i[1:], i[:-1]]), symmetric=False)
        src, dst = np.repeat(i, np.diff(both[0])), both[1]
        keep = (src < dst) | (src % 37 != 0)
        return shuffled(wl.csr_from_edges(n, src[keep], dst[keep], symmetric=False), seed)
    if kind == "two hubs":                   # a path whose middle part hangs on two vertices with more edges than are searched for a reverse
        m, leaves = n // 2, np.arange(100)
        src = np.concatenate([i[:m - 1], np.full(100, m // 2), np.full(100, m // 2 + 1)])
        dst = np.concatenate([i[1:m], m + leaves, m + 100 + leaves])
        return shuffled(wl.csr_from_edges(n, src, dst, symmetric=True), seed)
    side = int(n ** 0.5)                     # a grid whose edges lead right and down
    v = np.arange(side * side).reshape(side, side)
    return shuffled(wl.csr_from_edges(n, np.concatenate([v[:, :-1].ravel(), v[:-1].ravel()]), np.concatenate([v[:, 1:].ravel(), v[1:].ravel()]),
                                      symmetric=False), seed)


KINDS = ("ring", "directed ring", "one way", "two hubs", "grid")


@pytest.mark.parametrize("total,D", [(9000, 1), (25000, 6), (48000, 40)])       # rows of 32, 64 and 128 targets
def test_long_ways_in_a_batch(total, D):
    graphs, at = [], 0
    while sum(len(g[0]) - 1 for g in graphs) < total:
        graphs.append(long_ways(700 + 61 * at % 450, KINDS[at % len(KINDS)], at))
        at += 1
    check(wl.Workload("far", wl.pack_graphs(graphs), 1, 32, D))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [3300, 6100, 14300])       # edge list in shared memory; in the workspace, two blocks per SM and one
def test_long_ways_in_one_graph(n, kind):
    one(long_ways(n, kind, n), 5)
