"""Degenerate inputs and argument errors through the C ABI: batches that contain empty graphs, a
single-node batch, misaligned pointers, unsupported shapes.  Results against the oracle, errors by code."""
import numpy as np
import pytest
import torch

from oracle import attention as oattn
from oracle import spd as ospd
from paper_2609_34420_b200 import binding as gt
from paper_2609_34420_b200 import workloads as wl

from gpu_util import DeviceCase, gpu_spd, rel_l2, to_f64

pytestmark = pytest.mark.gpu


def test_packed_batch_with_empty_graphs_at_the_start_middle_and_end():
    graphs = [wl.erdos_renyi(n, 0.05, 3 + i) if n else (np.zeros(1, np.int32), np.zeros(0, np.int32))
              for i, n in enumerate([0, 70, 0, 0, 130, 1, 0])]
    w = wl.Workload("with_empty", wl.pack_graphs(graphs), 2, 64, 5, seed=3)
    bt = w.batch
    assert list(np.diff(bt.cu_seqlens)) == [0, 70, 0, 0, 130, 1, 0]
    got = gpu_spd(w).cpu().numpy()
    np.testing.assert_array_equal(got, ospd.spd_packed(bt.row_ptr, bt.col_idx, bt.cu_seqlens, w.max_dist))
    case = DeviceCase(w)
    out, lse = case.forward()
    dq, dk, dv, db = case.backward(out, lse)
    q, k, v, do, b = case.host_f64()
    ro, rl = oattn.forward_batch(q, k, v, case.spd_host, bt.spd_offsets, bt.cu_seqlens, b)
    ref = oattn.backward_batch(q, k, v, do, case.spd_host, bt.spd_offsets, bt.cu_seqlens, b)
    assert np.abs(to_f64(out) - ro).max() <= 1e-2 and np.abs(to_f64(lse) - rl).max() <= 1e-3
    for name, got_, want in zip(("dq", "dk", "dv", "dbias"), (dq, dk, dv, db), ref):
        assert rel_l2(to_f64(got_), want) <= 2e-2, name


def test_single_node_graph_attends_to_itself():
    w = wl.small_workload([1], 2, 32, 3, seed=1)
    case = DeviceCase(w)
    out, lse = case.forward()
    assert torch.equal(out, case.v)                         # softmax over one key: the output is its value row
    np.testing.assert_allclose(to_f64(lse)[:, 0],
                               (to_f64(case.q)[0] * to_f64(case.k)[0]).sum(-1) / np.sqrt(32.0) + to_f64(case.bias)[:, 0], atol=1e-3)
    dq, dk, dv, db = case.backward(out, lse)
    assert (to_f64(dq) == 0).all() and (to_f64(dk) == 0).all() and (to_f64(db) == 0).all()      # dS = P (dP - Delta) = 0
    assert torch.equal(dv, case.dout)


def _fwd_status(case, **over):
    a = dict(q=case.q, k=case.k, v=case.v, spd=case.spd, bias=case.bias, batch=case.batch, max_dist=case.w.max_dist,
             out=torch.empty_like(case.q), lse=torch.empty(case.H, case.T, device="cuda"))
    a.update(over)
    try:
        gt.gt_biased_attn_fwd(a["q"], a["k"], a["v"], a["spd"], a["bias"], a["batch"], a["max_dist"], a["out"], a["lse"])
    except gt.GtError as e:
        return e.status
    return 0


def test_argument_errors_are_codes_not_launches():
    case = DeviceCase(wl.small_workload([40], 2, 32, 5, seed=0))
    assert _fwd_status(case) == 0
    # a pointer that is not 16-byte aligned (TMA needs it): a view shifted by one bf16 element
    flat = torch.zeros(case.q.numel() + 8, dtype=torch.bfloat16, device="cuda")
    shifted = flat[1:1 + case.q.numel()].view_as(case.q)
    assert shifted.data_ptr() % 16 != 0
    assert _fwd_status(case, q=shifted) == 1                # GT_ERR_INVALID_ARG
    assert _fwd_status(case, max_dist=0) == 1 and _fwd_status(case, max_dist=255) == 1
    bad_batch = gt.Batch(n_total=40, n_graphs=2)            # two graphs without cu_seqlens / offsets
    assert _fwd_status(case, batch=bad_batch) == 1
    # head_dim outside {32, 64}
    x = torch.zeros(40, 2, 48, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(gt.GtError) as e:
        gt.gt_biased_attn_fwd(x, x, x, case.spd, case.bias, case.batch, 5, torch.empty_like(x), torch.empty(2, 40, device="cuda"))
    assert e.value.status == 2                              # GT_ERR_UNSUPPORTED
    # a workspace smaller than the query
    with pytest.raises(gt.GtError) as e:
        gt.gt_biased_attn_bwd(case.q, case.k, case.v, case.q, case.dout, torch.zeros(2, 40, device="cuda"), case.spd, case.bias,
                              case.batch, 5, *(torch.empty_like(case.q) for _ in range(3)), torch.empty_like(case.bias),
                              workspace=torch.zeros(512, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 3                              # GT_ERR_WORKSPACE
    torch.cuda.synchronize()


def shifted(t, by):
    """The same tensor, `by` elements behind an aligned address."""
    store = torch.zeros(t.numel() + by, dtype=t.dtype, device=t.device)
    view = store[by:].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("d", [32, 64])
@pytest.mark.parametrize("by", [1, 2])
def test_feature_attention_takes_tensors_at_any_element(d, by):
    n, H, dev = 150, 2, "cuda"
    gen = torch.Generator(device=dev).manual_seed(d + by)
    q, k, v, do = (torch.randn(n, H, d, device=dev, generator=gen).bfloat16() for _ in range(4))
    feat = torch.randint(0, 256, (n, n, 4), device=dev, generator=gen, dtype=torch.uint8)
    w = torch.randn(H, 4, device=dev, generator=gen) * 0.01

    def run(move):
        a = [move(x) for x in (q, k, v, do)]
        out, dq, dk, dv = (move(torch.full_like(q, float("nan"))) for _ in range(4))
        lse, dw = torch.empty(H, n, device=dev), torch.empty_like(w)
        gt.gt_feature_attn_fwd(a[0], a[1], a[2], feat, w, gt.Batch(n), out, lse)
        gt.gt_check(gt.gt_feature_attn_bwd(*a, lse, feat, w, gt.Batch(n), dq, dk, dv, dw))
        return out, lse, dq, dk, dv, dw

    for got, want in zip(run(lambda x: shifted(x, by)), run(lambda x: x)):
        assert torch.equal(got, want)
    odd = torch.zeros(2 * q.numel() + 1, dtype=torch.uint8, device=dev)[1:]            # refused on the host, nothing is launched
    st = gt.lib().gt_feature_attn_fwd(odd.data_ptr(), k.data_ptr(), v.data_ptr(), feat.data_ptr(), w.data_ptr(), gt.Batch(n)._c_pair()[1], H, d,
                                      q.data_ptr(), torch.empty(H, n, device=dev).data_ptr(), None)
    assert st == 1


def test_codes_are_written_at_any_address():
    n, dev = 37, "cuda"
    f = torch.randint(0, 3, (n, n, 4), device=dev, dtype=torch.uint8)
    vectors = torch.empty(256, dtype=torch.int32, device=dev)
    out = []
    for by in (0, 1, 2):
        codes = shifted(torch.full((n * 48,), 77, dtype=torch.uint8, device=dev), by)
        gt.gt_check(gt.gt_feature_encode(f, gt.Batch(n), codes, vectors))
        out.append(codes.clone())
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


@pytest.mark.parametrize("by", [1, 8, 18])
def test_distances_are_written_at_any_address(by):
    """A ragged batch of blocks of 128 targets with a ring that is finished by shortcuts, single graphs of both pull kernels; the bit
    matrices, which work on 16 bytes at a time, refuse it on the host."""
    from gpu_util import device_batch, device_csr
    i = np.arange(900)
    ring = wl.csr_from_edges(900, i, (i + 1) % 900, symmetric=True)
    wide = [wl.random_geometric(900 + 5 * j, 5.0, j) for j in range(42)] + [ring]
    for graphs in ([wl.erdos_renyi(70, 0.05, 3)], [ring], wide, [wl.erdos_renyi(6001, 0.0016, 4)]):
        b = wl.pack_graphs(graphs)
        bt = device_batch(b)
        rp, ci = device_csr(b)
        out = shifted(torch.full((b.spd_bytes,), 77, dtype=torch.uint8, device="cuda"), by)
        gt.gt_check(gt.gt_spd_build(rp, ci, bt, 6, out))
        np.testing.assert_array_equal(out.cpu().numpy(), ospd.spd_packed(b.row_ptr, b.col_idx, b.cu_seqlens, 6))
    b = wl.pack_graphs([wl.erdos_renyi(19000, 0.0001, 5)])
    rp, ci = device_csr(b)
    with pytest.raises(gt.GtError) as e:
        gt.gt_spd_build(rp, ci, device_batch(b), 6, shifted(torch.zeros(b.spd_bytes, dtype=torch.uint8, device="cuda"), by))
    assert e.value.status == 1
