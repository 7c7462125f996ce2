"""GPU parity of the training-side pieces against the oracle, through the C
ABI: the hidden-state alignment of Eq. 9 (value and gradient), the output
alignment of Eq. 10 (KL over the classes of an LM head), and the router's
gradient through the score gate (Sec. 3.4, differentiable score pathway)."""
import numpy as np
import pytest
import torch

from oracle import adadsf_oracle as O
from paper_2607_21291_gb300 import synth as S
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    from paper_2607_21291_gb300 import adadsf
    adadsf.lib()
    return adadsf


@pytest.mark.parametrize("n,d,dtype", [(1, 64, "f32"), (3001, 1024, "bf16"), (777, 512, "f32"), (40, 3584, "bf16")])
def test_align_hidden(A, n, d, dtype):
    g = np.random.default_rng(n + d)
    hs = S.round_to(g.standard_normal((n, d)).astype(np.float32) * 2, dtype)
    hd = S.round_to((hs + 0.5 * g.standard_normal((n, d))).astype(np.float32), dtype)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    grad = torch.empty((n, d), dtype=torch.float32, device="cuda")
    A.adadsf_align_hidden(H.to_dev(hs, td), H.to_dev(hd, td), acc, grad)
    got = acc.cpu().numpy()
    ref = O.hidden_alignment(hs.astype(np.float64), hd.astype(np.float64))
    assert got[1] == n
    assert got[0] == pytest.approx(ref.sum(), rel=1e-4)
    H.assert_close(grad.cpu().numpy(), O.hidden_alignment_grad(hs.astype(np.float64), hd.astype(np.float64)),
                   1e-3, "grad")
    again = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_align_hidden(H.to_dev(hs, td), H.to_dev(hd, td), again)
    assert again.cpu().numpy().tolist() == got.tolist()        # fixed summation order


@pytest.mark.parametrize("n,d,dtype,shift", [(9, 256, "bf16", 0), (33, 512, "bf16", 0), (17, 520, "bf16", 0),
                                              (70, 2056, "bf16", 0), (5, 4096, "bf16", 0), (5, 4104, "bf16", 0),
                                              (12, 2048, "f32", 0), (12, 250, "f32", 0), (31, 1000, "f32", 1),
                                              (20000, 64, "bf16", 0)])
def test_align_hidden_widths(A, n, d, dtype, shift):
    """Row widths on both sides of every register layout (one warp or 128
    threads a row, one to four vectors a thread) and of the general path (width
    not whole vectors, too wide, gradient at an odd float). Softmax sums of d
    fp32 terms: 2e-5 of the largest gradient element. An element p (r - p.r) / n
    carries a few 2^-24 of p whatever r - p.r leaves of it, and the largest p are
    up to a few thousand times the gradient's rms: under 1e-3 of the rms.
    Twice the same bits."""
    g = np.random.default_rng(n + d)
    hs = S.round_to(g.standard_normal((n, d)).astype(np.float32) * 2, dtype)
    hd = S.round_to((hs + 0.5 * g.standard_normal((n, d))).astype(np.float32), dtype)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    store = torch.full((n * d + 8,), 7.0, device="cuda")
    grad = store[shift:shift + n * d].view(n, d)
    A.adadsf_align_hidden(H.to_dev(hs, td), H.to_dev(hd, td), acc, grad)
    ref = O.hidden_alignment(hs.astype(np.float64), hd.astype(np.float64))
    assert acc.cpu().numpy()[0] == pytest.approx(ref.sum(), rel=1e-5) and float(acc[1]) == n
    H.assert_close(grad.cpu().numpy(), O.hidden_alignment_grad(hs.astype(np.float64), hd.astype(np.float64)), 2e-5,
                   "grad", elem_tol=1e-3)
    assert float(store[shift + n * d]) == 7.0                   # nothing past the last row
    again = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_align_hidden(H.to_dev(hs, td), H.to_dev(hd, td), again, grad)
    assert again.cpu().numpy().tolist() == acc.cpu().numpy().tolist()


@pytest.mark.parametrize("n,d,V,dtype", [(64, 1024, 2048, "bf16"), (5, 64, 128, "bf16"), (33, 512, 1000, "f32"),
                                         (300, 768, 6272, "bf16")])
def test_align_output(A, n, d, V, dtype):
    g = np.random.default_rng(n * V + d)
    hs = S.round_to(g.standard_normal((n, d)).astype(np.float32), dtype)
    hd = S.round_to((hs + 0.3 * g.standard_normal((n, d))).astype(np.float32), dtype)
    W = S.round_to((g.standard_normal((V, d)) * 0.05).astype(np.float32), dtype)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_align_output(H.to_dev(hs, td), H.to_dev(hd, td), H.to_dev(W, td), acc)
    got = acc.cpu().numpy()
    ref = O.output_alignment(hs.astype(np.float64), hd.astype(np.float64), W.astype(np.float64))
    assert got[1] == n
    assert got[0] == pytest.approx(ref.sum(), rel=2e-3)
    same = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_align_output(H.to_dev(hs, td), H.to_dev(hs, td), H.to_dev(W, td), same)
    assert abs(same.cpu().numpy()[0]) < 1e-5 * n                # KL(P || P) = 0


@pytest.mark.parametrize("n,d,V,scale", [(1, 64, 64, 1.0), (127, 64, 192, 4.0), (129, 128, 19456, 1.0),
                                          (300, 320, 25664, 3.0), (1300, 64, 64, 1.0)])
def test_align_output_tiles(A, n, d, V, scale):
    """bf16: rows and classes around the 128 x 128 tiles, row blocks that start
    inside a CTA's range of tiles, a last tile of 64 classes, and logits wide
    enough that the running maxima move. The logits are fp32 sums of exact
    products (a few 1e-6 relative), so the loss holds to 1e-4 of its value; twice
    the same bits."""
    g = np.random.default_rng(n + V)
    hs = S.round_to(g.standard_normal((n, d)).astype(np.float32), "bf16")
    hd = S.round_to((hs + 0.3 * g.standard_normal((n, d))).astype(np.float32), "bf16")
    W = S.round_to((g.standard_normal((V, d)) * scale / np.sqrt(d)).astype(np.float32), "bf16")
    args = [H.to_dev(a, torch.bfloat16) for a in (hs, hd, W)]
    ws = A.workspace(A.lib().adadsf_align_workspace_size(n, V))
    vals = []
    for _ in range(2):
        acc = torch.zeros(2, dtype=torch.float64, device="cuda")
        A.adadsf_align_output(*args, acc, ws=ws)
        assert A.adadsf_sync_check(ws) == A.OK
        vals.append(acc.cpu().numpy().tolist())
    ref = O.output_alignment(hs.astype(np.float64), hd.astype(np.float64), W.astype(np.float64))
    assert vals[0][1] == n and vals[0] == vals[1]
    assert vals[0][0] == pytest.approx(ref.sum(), rel=1e-4)


@pytest.mark.parametrize("at", [0, 32, 96, 128, 160])
@pytest.mark.parametrize("mask", ["student_inf", "student_lowest", "student_1e30", "both_lowest"])
def test_align_output_masked_classes(A, mask, at):
    """bf16: 32 classes masked by logits at the lowest finite value or past it
    (-inf, by overflow of the sum), at every place of a chunk in its tile. A class
    that the dense model allows and the student gives -inf makes the loss +inf (the
    student's lowest values too, or near 1e39: a row's fp32 sum of them may
    overflow); at -1e30 they dominate it, in both models at once they drop out.
    (fp32 sums: 1e-4 of the value, as for the tiles.)"""
    g = np.random.default_rng(at)
    n, d, V = 70, 64, 192
    lowest = float(torch.finfo(torch.bfloat16).min)
    hs = S.round_to(g.standard_normal((n, d)).astype(np.float32), "bf16")
    hd = S.round_to((hs + 0.3 * g.standard_normal((n, d))).astype(np.float32), "bf16")
    W = S.round_to((g.standard_normal((V, d)) / np.sqrt(d)).astype(np.float32), "bf16")
    W[:, 0] = 0.0
    W[at:at + 32] = 0.0
    W[at:at + 32, 0] = 2.0 if mask == "student_inf" else 1.0
    hs[:, 0] = S.round_to(np.float32([-1e30]), "bf16")[0] if mask == "student_1e30" else lowest
    hd[:, 0] = lowest if mask == "both_lowest" else 0.0
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    ws = A.workspace(A.lib().adadsf_align_workspace_size(n, V))
    A.adadsf_align_output(*(H.to_dev(a, torch.bfloat16) for a in (hs, hd, W)), acc, ws=ws)
    assert A.adadsf_sync_check(ws) == A.OK
    got = float(acc[0])
    if mask in ("student_inf", "student_lowest"):
        assert got == np.inf if mask == "student_inf" else got > 1e37
        return
    ls, ld = (h.astype(np.float64) @ W.astype(np.float64).T for h in (hs, hd))
    lse = lambda l: l.max(1, keepdims=True) + np.log(np.exp(l - l.max(1, keepdims=True)).sum(1, keepdims=True))
    lps, lpd = ls - lse(ls), ld - lse(ld)
    ref = float((np.exp(lpd) * (lpd - lps)).sum())
    assert np.isfinite(got) and got == pytest.approx(ref, rel=1e-4)


def test_align_output_many_row_blocks(A):
    """bf16, 64 classes: a tile a row block, and more than two row blocks for
    every CTA of the persistent grid. Loss of each quarter of the rows against its
    own call."""
    n = 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + 200
    n -= n % 4
    g = torch.Generator(device="cuda").manual_seed(n)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    hd = rnd(n, 64)
    hs, hd, W = (hd + 0.3 * rnd(n, 64)).bfloat16(), hd.bfloat16(), (rnd(64, 64) / 8).bfloat16()
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    ws = A.workspace(A.lib().adadsf_align_workspace_size(n, 64))
    A.adadsf_align_output(hs, hd, W, acc, ws=ws)
    assert A.adadsf_sync_check(ws) == A.OK
    ls, ld = (torch.log_softmax(h.double() @ W.double().T, -1) for h in (hs, hd))
    ref = (ld.exp() * (ld - ls)).sum().item()
    assert acc[1].item() == n and acc[0].item() == pytest.approx(ref, rel=1e-5)


QWEN_SMALL = S.QWEN25_1_5B.replace(d=1024, n_heads=8, n_kv_heads=2, ffn=1536, n_layers=1)


@pytest.mark.parametrize("shape,B,T,K", [(QWEN_SMALL, 2, 150, 70), (S.PYTHIA_160M.replace(n_layers=1), 3, 100, 37),
                                         (S.PYTHIA_70M.replace(n_layers=1), 1, 128, 64),
                                         (QWEN_SMALL, 2, 2048, 1500)])
def test_router_backward(A, shape, B, T, K):
    """The gated layer on the GPU, the ungated one on the same kept set (its
    delta), an upstream gradient G; the router gradient matches the oracle's
    chain rule on the same delta, and the gated layer still matches the
    oracle's gated layer."""
    td = H.tdtype(shape)
    W = H.host_layer(shape, 41)
    x = S.round_to(S.hidden(41, B, T, shape.d), shape.dtype)
    wd = A.to_device(W, td)
    outs = {}
    for flags in (A.FLAG_GATE_SIGMOID, 0):
        cfg = A.make_cfg(shape, flags)
        xd = H.to_dev(x, td)
        idx = torch.empty((B, K), dtype=torch.int32, device="cuda")
        ws = A.workspace(A.adadsf_layer_workspace_size(cfg, B, T, K))
        A.adadsf_sparse_layer_forward(cfg, wd, xd, K, idx, None, ws)
        assert A.adadsf_sync_check(ws) == A.OK
        outs[flags] = (xd, idx)
    (yg, idx_g), (yp, idx_p) = outs[A.FLAG_GATE_SIGMOID], outs[0]
    assert torch.equal(idx_g, idx_p)
    gi = idx_g.cpu().numpy()
    rows = (np.arange(B)[:, None] * T + gi).reshape(-1)
    G = np.random.default_rng(B * T + K).standard_normal((B * T, shape.d)).astype(np.float32)
    grad = A.adadsf_router_backward(A.make_cfg(shape, A.FLAG_GATE_SIGMOID), wd, H.to_dev(x, td), yp,
                                    torch.from_numpy(rows.astype(np.int32)).cuda(), H.to_dev(G, torch.float32))
    x64 = x.astype(np.float64)
    delta = (H.to_np(yp).reshape(-1, shape.d) - x64.reshape(-1, shape.d))[rows]
    ref = O.router_grad(x64, H.f64(W), rows, delta, G.astype(np.float64)[rows])
    h, d = shape.router_hidden, shape.d
    g = grad.cpu().numpy().astype(np.float64)
    parts = {"router_w1": g[:h * d].reshape(h, d), "router_b1": g[h * d:h * d + h],
             "router_w2": g[h * d + h:h * d + 2 * h], "router_b2": g[h * d + 2 * h:]}
    tol = 2e-3 if shape.dtype == "bf16" else 1e-4
    for k, v in parts.items():
        H.assert_close(v, ref[k], tol, k)
    # and the gated forward itself follows the oracle's gated layer
    refg, _, _ = O.sparse_layer_forward(x64, H.f64(W), dict(O.params_of(shape), gate="sigmoid"), K, idx=gi)
    H.assert_close(H.to_np(yg), refg, H.tol(shape), "gated layer")


@pytest.mark.parametrize("n,d,h,dtype,shift", [(1, 64, 64, "bf16", 0), (15, 192, 40, "f32", 1), (17, 4096, 64, "bf16", 0),
                                              (263, 2048, 64, "f32", 0), (1000, 320, 64, "bf16", 1),
                                              (33, 64, 3, "f32", 0)])
def test_router_backward_edges(A, n, d, h, dtype, shift):
    """Kept counts around the 16-row blocks and the eighths of the reduction,
    feature widths that are not multiples of its 64 columns times the warps,
    few hidden units, kept rows in any order, and an upstream gradient at an
    odd float. Same inputs on both sides, so only fp32 sums differ: about
    sqrt(d) + sqrt(n) roundings of 2^-24 each (under 1e-5 of the largest
    element at these sizes)."""
    shape = S.PYTHIA_70M.replace(d=d, router_hidden=h, n_layers=1, dtype=dtype)
    td = H.tdtype(shape)
    W = H.host_layer(shape, n + d)
    BT = n + 37
    x = S.round_to(S.hidden(n, 1, BT, d), dtype)
    y = S.round_to(x + 0.3 * S.hidden(n + 1, 1, BT, d), dtype)
    g = np.random.default_rng(n * d)
    G = g.standard_normal((BT, d)).astype(np.float32)
    rows = g.permutation(BT)[:n].astype(np.int32)
    store = torch.empty(BT * d + 4, dtype=torch.float32, device="cuda")
    Gd = store[shift:shift + BT * d].view(BT, d)
    Gd.copy_(torch.from_numpy(G))
    got = A.adadsf_router_backward(A.make_cfg(shape, A.FLAG_GATE_SIGMOID), A.to_device(W, td), H.to_dev(x, td),
                                   H.to_dev(y, td), torch.from_numpy(rows).cuda(), Gd).cpu().numpy().astype(np.float64)
    x64 = x.astype(np.float64)
    delta = (y.astype(np.float64) - x64).reshape(BT, d)[rows]
    ref = O.router_grad(x64, H.f64(W), rows, delta, G.astype(np.float64)[rows])
    parts = {"router_w1": got[:h * d].reshape(h, d), "router_b1": got[h * d:h * d + h],
             "router_w2": got[h * d + h:h * d + 2 * h], "router_b2": got[h * d + 2 * h:]}
    for k, v in parts.items():
        H.assert_close(v, ref[k], 2e-5, k)


@pytest.mark.parametrize("shape,lr", [(S.PYTHIA_70M.replace(n_layers=1), 3000.0),
                                      (QWEN_SMALL.replace(dtype="f32"), 3000.0)])
def test_router_alignment_descends(A, shape, lr):
    """Plain SGD on the router through the gated layer (paper_2607_21291_gb300.align)
    lowers the layer's Eq. 9 loss against the dense layer's output: the
    gradient points downhill."""
    from paper_2607_21291_gb300 import align
    B, T, K = 2, 96, 48
    td = H.tdtype(shape)
    w = A.to_device(H.host_layer(shape, 51), td)
    x = H.to_dev(S.round_to(S.hidden(51, B, T, shape.d), shape.dtype), td)
    cfg = A.make_cfg(shape)
    h_dense = x.clone()
    A.adadsf_sparse_layer_forward(cfg, w, h_dense, T)          # the dense layer
    losses = [align.router_alignment_step(cfg, w, x, h_dense, K, lr) for _ in range(6)]
    # the first step goes downhill and the loss stays below its start (with a
    # fixed step size it may settle and wander slightly near its floor)
    assert losses[1] < losses[0] * 0.999, losses
    assert max(losses[1:]) < losses[0], losses
