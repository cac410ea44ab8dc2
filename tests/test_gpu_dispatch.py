"""The edges of the size rules by which the attention kernels choose their form, against the fp64 oracle
(tolerances of the forward and backward parity tests, whose checks these call)."""
import numpy as np
import pytest
import torch

from oracle import attention as oattn
from paper_2609_34420_b200 import binding as gt
from paper_2609_34420_b200 import workloads as wl

from gpu_util import DeviceCase, rel_l2, to_f64
from test_gpu_attn_bwd import check_backward
from test_gpu_attn_fwd import LSE_MAX_ABS, check_forward, oracle_forward, pytestmark  # noqa: F401  (GPU tests)


def sizes(n_graphs, largest):
    """One graph that dominates the grid of a batch; the others end at, before and behind the edges of 128 and 256 rows."""
    rest = [1, 127, 128, 129, 255, 256, 257, 16, 300, 31]
    return ([rest[i % len(rest)] for i in range(n_graphs // 2)] + [largest] + [rest[-1 - i % len(rest)] for i in range(n_graphs - n_graphs // 2 - 1)])


# up to 64 graphs the work list is sorted, beyond that in batch order; 2 graphs: no list in the forward
@pytest.mark.parametrize("n_graphs,largest,d", [(2, 257, 64), (40, 1500, 32), (64, 1281, 64), (65, 1281, 32), (97, 1024, 64)])
def test_packed_batches_with_and_without_a_work_list(n_graphs, largest, d):
    case, out, lse = check_forward(wl.small_workload(sizes(n_graphs, largest), 4, d, 6, seed=n_graphs, avg_degree=1.8))
    # a workspace of the header alone: no tensor maps, no list, the SPD tiles come by 16-byte copies; same arithmetic
    ws = torch.zeros(256, dtype=torch.uint8, device=case.q.device)
    out2, lse2 = torch.full_like(out, float("nan")), torch.full_like(lse, float("nan"))
    gt.gt_biased_attn_fwd(case.q, case.k, case.v, case.spd, case.bias, case.batch, case.w.max_dist, out2, lse2, ws)
    gt.gt_check(ws)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


# up to 1 152 nodes two blocks of one query tile share an SM, if the workspace has room for their list; else blocks of two tiles
@pytest.mark.parametrize("largest,d,D", [(1152, 64, 6), (1153, 64, 6), (1152, 32, 40), (1100, 64, 40)])
def test_packed_batches_of_small_graphs(largest, d, D):
    w = wl.small_workload([largest, 1, 128, 129, 255, 256, 257] + sizes(12, largest), 4, d, D, seed=largest + D, avg_degree=1.8)
    case, out, lse = check_forward(w)
    _, _, out32 = case.forward_ex()
    assert rel_l2(to_f64(out32), oracle_forward(case)[0]) <= 1e-4        # as for the precise forward below
    need = gt.gt_biased_attn_fwd_workspace(case.batch, case.w.n_heads, d)
    for size in (need - 1, 256):
        ws = torch.zeros(size, dtype=torch.uint8, device=case.q.device)
        out2, lse2 = torch.full_like(out, float("nan")), torch.full_like(lse, float("nan"))
        gt.gt_biased_attn_fwd(case.q, case.k, case.v, case.spd, case.bias, case.batch, D, out2, lse2, ws)
        gt.gt_check(ws)
        assert torch.equal(out, out2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("n_graphs,largest,d", [(2, 129, 32), (64, 700, 64), (65, 700, 32)])
def test_packed_backward_work_list(n_graphs, largest, d):
    check_backward(wl.small_workload(sizes(n_graphs, largest), 2, d, 6, seed=n_graphs, avg_degree=1.8))


# private bin columns up to 26 buckets, then half as many columns per bucket at every doubling
@pytest.mark.parametrize("buckets", [26, 27, 52, 53, 104, 105, 208, 209, 256])
def test_bias_gradient_at_the_edges_of_the_bin_columns(buckets):
    check_backward(wl.small_workload([260], 2, 64 if buckets % 2 else 32, buckets - 2, seed=buckets, avg_degree=1.1))


def test_bias_gradient_reaches_every_bucket_of_a_path():
    n, D = 400, 120
    i = np.arange(n - 1)
    w = wl.small_workload([n], 2, 64, D, seed=1)
    w.batch = wl.pack_graphs([wl.csr_from_edges(n, i, i + 1, symmetric=True)])
    check_backward(w)


# 512 nodes: every tile takes its maximum first; beyond that only the tiles whose scores may be out of reach of the row's
# reference.  Inputs of 3 standard deviations and wide bias tables put some rows on either side.
@pytest.mark.parametrize("sizes_,d,D,std,spread", [([512], 64, 5, 1.0, 1.0), ([513], 32, 5, 1.0, 1.0), ([1100], 64, 60, 2.0, 12.0),
                                                   ([1100], 64, 20, 3.0, 1.0), ([900], 32, 254, 3.0, 30.0), ([700, 3, 1300, 256], 64, 9, 3.0, 4.0)])
def test_precise_forward_with_tiles_in_and_out_of_reach(sizes_, d, D, std, spread):
    w = wl.small_workload(sizes_, 2, d, D, seed=sum(sizes_) + D, avg_degree=1.3, qkv_std=std)
    w.tensors().bias[:] *= spread
    case = DeviceCase(w)
    out, lse, out32 = case.forward_ex()
    ro, rl = oracle_forward(case)
    # two bf16 terms of P: 2^-17 of each entry; scores of up to 100 in fp32: 100 * 2^-22 of each entry
    assert rel_l2(to_f64(out32), ro) <= 1e-4 and np.abs(to_f64(lse) - rl).max() <= LSE_MAX_ABS
    ws = torch.zeros(256, dtype=torch.uint8, device=case.q.device)       # no room for the norms: maximum first everywhere
    out32b = torch.full_like(out32, float("nan"))
    gt.gt_biased_attn_fwd_ex(case.q, case.k, case.v, case.spd, case.bias, case.batch, w.max_dist, out, lse, out32b, ws)
    gt.gt_check(ws)
    assert rel_l2(to_f64(out32b), ro) <= 1e-4


# one 128-row query tile per thread block up to 148 of them, two beyond: ragged graphs on either side of the line
@pytest.mark.parametrize("n", [128, 257, 300, 513])
@pytest.mark.parametrize("beyond", [0, 1])
def test_one_and_two_query_tiles_per_block(n, beyond):
    tiles = -(-n // 128)
    check_forward(wl.small_workload([n], 148 // tiles + beyond, 32 if n % 2 else 64, 5, seed=n + beyond, avg_degree=2.0))


# a key tile's queries shared by a cluster of 2, 3 or 4 blocks (private and shared bins), batches without a work list whose last graph
# has fewer tiles than the cluster has blocks (two and three blocks leave at once), one that takes the list, and the first size without
@pytest.mark.parametrize("sizes_,heads,d,D", [([385], 37, 32, 6), ([513], 7, 64, 6), ([640], 9, 64, 6), ([641], 8, 32, 24), ([900], 9, 64, 6),
                                              ([129], 2, 64, 60), ([300], 4, 32, 254), ([500, 500, 500], 2, 64, 9), ([512, 512, 256], 2, 64, 9),
                                              ([512, 512, 128], 2, 32, 40), ([512, 1], 4, 32, 9),
                                              ([3000], 8, 32, 6)])       # (the last: 192 blocks, two waves or three of shares)
def test_backward_with_shared_key_tiles(sizes_, heads, d, D):
    check_backward(wl.small_workload(sizes_, heads, d, D, seed=sum(sizes_) + D, avg_degree=2.0))


@pytest.mark.parametrize("chunks", [1, 3])
def test_chunked_backward_with_shared_key_tiles(chunks):
    w = wl.small_workload([700], 4, 64, 6, seed=chunks, avg_degree=2.0, directed=True)
    case, _ = check_backward(w)
    out, lse = case.forward()
    whole = case.backward(out, lse)
    for got, want in zip(case.backward_chunked(out, lse, chunks)[:4], whole):       # sums in another order, results rounded to bf16
        assert rel_l2(to_f64(got), to_f64(want)) <= 5e-3


# a query tile's keys shared by a cluster of 2, 3 or 4 blocks: the first size with it, shares of 3 tiles by which the last block has
# fewer, one key in the last tile, graphs of a batch with fewer tiles than blocks, wide bias tables (shares of different references)
@pytest.mark.parametrize("sizes_,heads,d,D,spread", [([641], 4, 64, 6, 1.0), ([700], 4, 32, 6, 12.0), ([1200], 3, 64, 60, 12.0), ([1025], 5, 64, 20, 1.0),
                                                     ([1100], 7, 32, 6, 12.0), ([800, 1, 300], 2, 64, 6, 1.0)])
def test_forward_with_shared_query_tiles(sizes_, heads, d, D, spread):
    w = wl.small_workload(sizes_, heads, d, D, seed=sum(sizes_) + D, avg_degree=1.5)
    w.tensors().bias[:] *= spread
    case, out, lse = check_forward(w)
    out_p, lse_p, out32 = case.forward_ex()
    ro, _ = oracle_forward(case)
    assert rel_l2(to_f64(out32), ro) <= 1e-4 and (lse_p - lse).abs().max().item() <= LSE_MAX_ABS


def test_backward_of_a_large_graph_among_many_of_one_node():
    """32 769 graphs whose largest has 256 x 256 tiles to transpose: a block for every tile of the largest graph and every graph
    would be more than a grid holds.  The large graph's gradients are those of the graph by itself (sums of dQ in another order,
    results rounded to bf16); a single node passes dout on to dv and has no other gradient."""
    n, G, before, d, D, dev = 32768, 32769, 20000, 32, 6, "cuda"
    lengths = np.ones(G, np.int64)
    lengths[before] = n
    cu = np.concatenate([[0], np.cumsum(lengths)])
    sizes_ = lengths * ((lengths + 15) // 16 * 16)
    off = np.concatenate([[0], np.cumsum(sizes_)])
    T = int(cu[-1])
    gen = torch.Generator(device=dev).manual_seed(5)
    q, k, v, do = (torch.randn(T, 1, d, device=dev, generator=gen).bfloat16() for _ in range(4))
    spd = torch.randint(0, D + 2, (int(off[-1]),), device=dev, generator=gen, dtype=torch.uint8)
    bias = torch.randn(1, D + 2, device=dev, generator=gen)

    def run(batch, q, k, v, do, spd):
        out, lse = torch.empty_like(q), torch.empty(1, q.shape[0], device=dev)
        gt.gt_check(gt.gt_biased_attn_fwd(q, k, v, spd, bias, batch, D, out, lse))
        grads = [torch.full_like(q, float("nan")) for _ in range(3)] + [torch.full_like(bias, float("nan"))]
        gt.gt_check(gt.gt_biased_attn_bwd(q, k, v, out, do, lse, spd, bias, batch, D, *grads))
        return [out] + grads

    packed = gt.Batch(T, G, n, torch.tensor(cu, dtype=torch.int32, device=dev), torch.tensor(off[:-1], dtype=torch.int64, device=dev))
    big = slice(before, before + n)
    single = torch.cat([torch.arange(before), torch.arange(before + n, T)]).to(dev)
    _, dq, dk, dv, _ = run(packed, q, k, v, do, spd)
    # P of a single key is 1 up to its rounding to bf16 (2^-9), and so are out and dP - Delta relative to v and dP
    assert ((dv[single] - do[single]).abs() <= do[single].abs() * 2.0 ** -7).all()
    assert max(x[single].float().abs().max().item() for x in (dq, dk)) <= 2.0 ** -8 * 4 * d
    do[single] = 0                                         # (these residues would add up in dbias)
    out, dq, dk, dv, db = run(packed, q, k, v, do, spd)
    alone = run(gt.Batch(n), *(x[big].contiguous() for x in (q, k, v, do)), spd[int(off[before]):int(off[before + 1])].clone())
    for got, want in zip((out, dq, dk, dv), alone):
        assert rel_l2(to_f64(got[big]), to_f64(want)) <= 5e-3
    assert rel_l2(to_f64(db), to_f64(alone[4])) <= 1e-3
    assert all(not x[single].any() for x in (dq, dk, dv))


# The softmax reference starts at 0: scores far above and far below it, a first tile far below the others, a first tile masked out.
@pytest.mark.parametrize("n,shift,masked", [(300, 60.0, False), (300, -60.0, False), (129, -17.0, False), (700, 17.0, False), (300, 0.0, True), (520, -90.0, True)])
def test_scores_far_from_the_first_reference(n, shift, masked):
    w = wl.small_workload([n], 2, 64, 6, seed=n, avg_degree=1.2)
    w.tensors().bias[:] += shift
    if masked:                                   # unreachable pairs weigh nothing; vertex 0 .. 127 reach each other only
        w.tensors().bias[:, 7] = -1e30
    check_forward(w)


# The same in the other forms of the kernel, with the fp32 output (whose tiles cannot be done twice) and with the chunks' own lse.
FORMS = {"one query tile": ([700], 2), "two query tiles": ([1100], 20), "two blocks per SM": (sizes(40, 500), 4)}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("shift,masked", [(60.0, False), (-60.0, False), (-90.0, False), (0.0, True), (-90.0, True)])
def test_scores_far_from_the_first_reference_in_every_form(form, shift, masked):
    sizes_, heads = FORMS[form]
    w = wl.small_workload(sizes_, heads, 64, 6, seed=heads, avg_degree=1.2)
    w.tensors().bias[:] += shift
    if masked:
        w.tensors().bias[:, 7] = -1e30
    case = DeviceCase(w)
    out, lse = case.forward()
    _, lse32, out32 = case.forward_ex()
    ro, rl = oracle_forward(case)
    # bf16 rounds each P and the result by up to 2^-8 of it (a masked row may be left with two nodes whose values nearly cancel)
    q, k, v, _, b = case.host_f64()
    weight, _ = oattn.forward_batch(q, k, np.abs(v), case.spd_host, w.batch.spd_offsets, w.batch.cu_seqlens, b)
    assert (np.abs(to_f64(out) - ro) <= 2.0 ** -8 * (weight + np.abs(ro)) + 1e-4).all()
    assert rel_l2(to_f64(out32), ro) <= 1e-4
    assert max(np.abs(to_f64(x) - rl).max() for x in (lse, lse32)) <= LSE_MAX_ABS
    if len(sizes_) == 1:
        for own in (True, False):
            oc, lc, _ = case.forward_chunked(5, want_chunk_lse=own)
            assert np.abs(to_f64(lc) - rl).max() <= LSE_MAX_ABS and rel_l2(to_f64(oc), to_f64(out)) <= 1e-3


# Without the chunks' own lse, on 148 SMs: each chunk in blocks of its own, all behind one another in blocks of one query tile and of
# two, and two or three behind one another (the last share as long, shorter, a single chunk).  Every chunk is a sum of its own in all
# of them and is added in fp32: beside the results with the chunks' own lse only values next to a tie of bf16 differ (relative
# differences of about 2^-21 move one in a few thousand by 2^-8), and lse is rounded once more or less (rms 2^-20 / sqrt(12) at 8 to 16).
@pytest.mark.parametrize("n,heads,d,chunks", [(1000, 4, 64, 3), (5000, 4, 64, 5), (10000, 4, 32, 2), (300, 2, 32, 2), (2048, 8, 64, 8), (9000, 4, 64, 8),
                                              (5537, 4, 64, 6), (6000, 4, 64, 8), (5300, 8, 32, 7), (65536, 4, 32, 8)])
def test_chunked_forward_in_parts(n, heads, d, chunks):
    dev, gen = torch.device("cuda"), torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(n, heads, d, device=dev, generator=gen).bfloat16() for _ in range(3))
    spd = torch.randint(0, 8, (n * wl.round_up(n, 16),), device=dev, generator=gen, dtype=torch.uint8)
    bias = torch.randn(heads, 8, device=dev, generator=gen)
    batch = gt.Batch(n)
    out, out_c, lse, lse_c = torch.empty_like(q), torch.empty_like(q), torch.empty(heads, n, device=dev), torch.empty(heads, n, device=dev)
    gt.gt_check(gt.gt_biased_attn_fwd_chunked(q, k, v, spd, bias, batch, 6, out, lse, chunks, torch.empty(chunks, heads, n, device=dev)))
    gt.gt_check(gt.gt_biased_attn_fwd_chunked(q, k, v, spd, bias, batch, 6, out_c, lse_c, chunks))
    assert rel_l2(to_f64(out_c), to_f64(out)) <= 1e-4
    assert (lse - lse_c).abs().max().item() <= LSE_MAX_ABS
    rows = torch.randperm(n, device=dev, generator=gen)[:256]
    pairs = spd.view(n, -1)[rows, :n].long()
    for h in range(heads):
        s = q[rows, h].double() @ k[:, h].double().T / d ** 0.5 + bias[h].double()[pairs]
        exact_lse = torch.logsumexp(s, 1)
        assert (lse_c[h, rows] - exact_lse).square().mean().sqrt().item() <= 4e-7
        assert rel_l2(to_f64(out_c[rows, h]), ((s - exact_lse[:, None]).exp() @ v[:, h].double()).cpu().numpy()) <= 5e-3


# References that move from chunk to chunk: the sums so far are brought to the new one.
@pytest.mark.parametrize("n,heads,chunks", [(2048, 8, 8), (9000, 4, 8), (5537, 4, 6)])
def test_chunked_forward_with_rising_scores(n, heads, chunks):
    dev, gen = torch.device("cuda"), torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(n, heads, 64, device=dev, generator=gen).bfloat16() for _ in range(3))
    j = torch.arange(wl.round_up(n, 16), device=dev) * 8 // n                # bucket 0: masked for every other row
    spd = torch.where(torch.arange(n, device=dev)[:, None] % 2 == 0, j, 7 - j.clamp(max=7)).clamp(max=7).to(torch.uint8)
    bias = 30.0 * torch.arange(8, device=dev, dtype=torch.float32).repeat(heads, 1) - 60.0
    bias[:, 0] = -1e30
    batch = gt.Batch(n)
    out, lse = torch.empty_like(q), torch.empty(heads, n, device=dev)
    gt.gt_check(gt.gt_biased_attn_fwd_chunked(q, k, v, spd.reshape(-1), bias, batch, 6, out, lse, chunks))
    rows = torch.randperm(n, device=dev, generator=gen)[:256]
    for h in range(heads):
        s = q[rows, h].double() @ k[:, h].double().T / 8 + bias[h].double()[spd[rows, :n].long()]
        exact_lse = torch.logsumexp(s, 1)
        assert (lse[h, rows] - exact_lse).abs().max().item() <= LSE_MAX_ABS
        assert rel_l2(to_f64(out[rows, h]), ((s - exact_lse[:, None]).exp() @ v[:, h].double()).cpu().numpy()) <= 5e-3
