"""gt_spd_build for one large graph, where only a core of its targets is searched for: bit-exact against the BFS oracle."""
import numpy as np
import pytest
import torch

from oracle import spd as ospd
from paper_2609_34420_b200 import binding as gt
from paper_2609_34420_b200 import workloads as wl

from gpu_util import device_batch, device_csr
from test_gpu_spd import check, pytestmark  # noqa: F401  (GPU tests)


def edges(csr):
    return np.repeat(np.arange(len(csr[0]) - 1), np.diff(csr[0])), csr[1]


def power_law(n, degree, tail=0, keep=1.0):
    """A power-law graph, every edge's two directions kept with probability `keep`, and a path of `tail` vertices behind vertex 0."""
    src, dst = edges(wl.chung_lu_power_law(n - tail, float(degree), 2.1, n))
    if keep < 1.0:
        kept = np.random.Generator(np.random.PCG64(n)).random(len(src)) < keep
        src, dst = src[kept], dst[kept]
    return with_tail(n, src, dst, tail)


def with_tail(n, src, dst, tail):
    t = np.arange(n - tail, n)
    back = np.concatenate([[0], t[:-1]])[:tail]
    return wl.csr_from_edges(n, np.concatenate([src, back, t]), np.concatenate([dst, t, back]), symmetric=False)


def tree(n):
    """A random recursive tree: dozens of levels, and more than half of its vertices are leaves or next to one."""
    i = np.arange(1, n)
    return wl.csr_from_edges(n, i, (np.random.Generator(np.random.PCG64(n)).random(n - 1) * i).astype(np.int64))


def star(n, inward):
    i, hub = np.arange(1, n), np.zeros(n - 1, np.int64)
    return wl.csr_from_edges(n, i, hub, symmetric=False) if inward else wl.csr_from_edges(n, hub, i)


GRAPHS = {
    "a plane for every level": (lambda: power_law(32768, 14), 24),
    "sources and columns ragged, distances clipped": (lambda: power_law(32775, 8), 4),
    "clipped just where four bits end": (lambda: power_law(32901, 6), 14),
    "directed": (lambda: power_law(33003, 8, keep=0.6), 254),
    # eleven levels have a plane of their own: five to six levels and the path's
    "levels that wait in the matrix": (lambda: with_tail(32777, *edges(wl.barabasi_albert(32770, 5, 3)), 7), 40),
    "more levels than four bits hold in one column block only": (lambda: power_law(33000, 8, tail=20), 17),
    # at every level nearly every row gains something
    "many rows in the matrix when the levels end": (lambda: wl.random_geometric(32769, 4.0, 1), 12),
    "a tree": (lambda: tree(32800), 30),
    "a core of one": (lambda: star(32770, False), 3),
    "in-neighbours only": (lambda: star(32772, True), 1),
    "no edges: no core": (lambda: wl.csr_from_edges(32768, np.zeros(0, np.int64), np.zeros(0, np.int64)), 5),
}


@pytest.mark.parametrize("name", GRAPHS)
def test_targets_that_follow_from_others(name):
    make, D = GRAPHS[name]
    check(wl.Workload("core", wl.pack_graphs([make()]), 1, 32, D))


# Five column blocks at a time (beyond 46 811 vertices there may be so many), five or six planes of frontiers: the levels behind those wait
# in the matrix, up to eight of them, and deeper blocks end in bytes. 
LARGE = {
    "some levels in the matrix": (lambda: with_tail(60000, *edges(wl.barabasi_albert(59993, 5, 3)), 7), 40),
    "all that fit in the matrix": (lambda: wl.erdos_renyi(60000, 6.0 / 60000, 4), 11),
    "deep, all vertices that 16 bits number": (lambda: power_law(65536, 18, tail=20), 24),
    "directed": (lambda: power_law(65536, 20, tail=9, keep=0.7), 254),
}


@pytest.mark.parametrize("name", LARGE)
def test_targets_that_follow_from_others_in_five_blocks(name):
    make, D = LARGE[name]
    csr = make()
    n = len(csr[0]) - 1
    b = wl.pack_graphs([csr])
    batch, (rp, ci) = device_batch(b, "cuda"), device_csr(b, "cuda")
    size = gt.gt_spd_build_workspace(batch, len(b.col_idx), D)
    got, every = (torch.full((b.spd_bytes,), 0xEE, dtype=torch.uint8, device="cuda") for _ in range(2))
    for out, room in ((got, size), (every, size - 1)):                       # (the smaller workspace: every target is searched for)
        ws = torch.zeros(room, dtype=torch.uint8, device="cuda")
        gt.gt_spd_build(rp, ci, batch, D, out, ws)
        gt.gt_check(ws)
        del ws
    assert torch.equal(got, every)
    rows = np.unique(np.concatenate([np.arange(16), np.arange(n - 32, n), np.random.default_rng(n).choice(n, 200, replace=False)]))
    ref = ospd.spd_rows(b.row_ptr, b.col_idx, D, rows)
    np.testing.assert_array_equal(got.view(n, -1)[torch.from_numpy(rows).cuda()].cpu().numpy(), ref)


def test_workspace_without_room_for_the_core():
    w = wl.Workload("core", wl.pack_graphs([power_law(32777, 8)]), 1, 32, 9)
    exp = check(w)
    batch, (rp, ci) = device_batch(w.batch, "cuda"), device_csr(w.batch, "cuda")
    ws = torch.zeros(gt.gt_spd_build_workspace(batch, len(w.batch.col_idx), w.max_dist) - 1, dtype=torch.uint8, device="cuda")
    out = torch.full((w.batch.spd_bytes,), 0xEE, dtype=torch.uint8, device="cuda")
    gt.gt_spd_build(rp, ci, batch, w.max_dist, out, ws)
    gt.gt_check(ws)
    np.testing.assert_array_equal(out.cpu().numpy(), exp)
