"""GPU parity of the individual steps against the fp64 oracle, through the C ABI.
Sizes span several tiles with ragged tails; edge cases include K = 0, 1, T-1, T,
ties, NaN and signed zeros."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from oracle import adadsf_oracle as O
from paper_2607_21291_gb300 import synth as S
from tests import helpers as H

pytestmark = pytest.mark.gpu
SYNC_BYTES = 16384   # arrival counters right after the device error word


@pytest.fixture(scope="module")
def A():
    from paper_2607_21291_gb300 import adadsf
    adadsf.lib()
    torch.cuda.init()
    return adadsf


# ---------------------------------------------------------------- failure channel
def test_bounded_wait_gives_up_cleanly(A):
    ws = A.workspace(256)
    A.adadsf_selftest_bounded_wait(ws, 2000)
    assert A.adadsf_sync_check(ws) == A.ERR_DEVICE_TIMEOUT
    assert A.adadsf_sync_check(ws) == A.OK              # cleared by the read
    x = torch.ones(16, device="cuda")
    assert float((x * 2).sum()) == 32.0                 # context still usable



def test_timeout_clears_sync_area(A):
    """A kernel that gives up waiting may leave cross-CTA arrival counters
    part-way. After a timeout, adadsf_sync_check zeroes the synchronisation
    area, so the same workspace then gives correct router scores on a shape
    whose tiles are split along d (counters in use)."""
    shape = S.QWEN25_7B.replace(ffn=256)
    n = 25600 - 77                                          # 200 tiles: split past one wave
    cfg = A.make_cfg(shape)
    ws = A.workspace(A.adadsf_router_select_workspace_size(cfg, 1, 1))
    ws[256:256 + SYNC_BYTES].view(torch.int32)[::7] = 3     # counters left part-way
    A.adadsf_selftest_bounded_wait(ws, 2000)
    assert A.adadsf_sync_check(ws) == A.ERR_DEVICE_TIMEOUT
    assert int(ws[256:256 + SYNC_BYTES].view(torch.int32).abs().sum()) == 0
    W = H.host_layer(shape, 3)
    x = S.round_to(np.random.default_rng(n + 1).standard_normal((n, shape.d)).astype(np.float32), shape.dtype)
    sc = torch.empty(n, dtype=torch.float32, device="cuda")
    A.adadsf_router_scores(cfg, A.to_device(W, H.tdtype(shape)), H.to_dev(x, H.tdtype(shape)), sc, ws=ws)
    assert A.adadsf_sync_check(ws) == A.OK
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    assert np.max(np.abs(sc.cpu().numpy() - ref)) / np.max(np.abs(ref)) < 5e-3

# ---------------------------------------------------------------- Top-K (Sec. 3.4)
@pytest.mark.parametrize("B,T,K", [(1, 1, 1), (3, 7, 3), (2, 128, 64), (4, 512, 256), (2, 1000, 1),
                                   (2, 1000, 999), (2, 1000, 1000), (5, 2048, 1024), (16, 4096, 2048),
                                   (1, 16384, 5000)])
def test_topk_random(A, B, T, K):
    g = np.random.default_rng(B * 100003 + T * 7 + K)
    s = g.standard_normal((B, T)).astype(np.float32)
    s[:, ::5] = np.round(s[:, ::5], 1)                 # plenty of exact ties
    sd = torch.from_numpy(s).cuda()
    idx = torch.full((B, K), -1, dtype=torch.int32, device="cuda")
    rows = torch.full((B, K), -1, dtype=torch.int32, device="cuda")
    A.adadsf_topk_select(sd, K, idx, rows)
    gi, gr = idx.cpu().numpy(), rows.cpu().numpy()
    for b in range(B):
        ref = O.topk_keep(s[b], K)
        assert gi[b].tolist() == ref.tolist()
        assert gr[b].tolist() == (b * T + ref).tolist()


def test_topk_special_values(A):
    s = np.array([[1.0, 3.0, 3.0, 2.0, 3.0, -0.0, 0.0, np.nan, -np.inf, np.inf, np.nan, -1.0]],
                 dtype=np.float32)
    sd = torch.from_numpy(s).cuda()
    for K in range(0, 13):
        idx = torch.full((1, max(K, 1)), -1, dtype=torch.int32, device="cuda")
        A.adadsf_topk_select(sd, K, idx)
        if K:
            assert idx[0].cpu().tolist() == O.topk_keep(s[0], K).tolist(), K
    allnan = torch.full((2, 33), float("nan"), device="cuda")
    idx = torch.empty((2, 5), dtype=torch.int32, device="cuda")
    A.adadsf_topk_select(allnan, 5, idx)
    assert idx.cpu().tolist() == [[0, 1, 2, 3, 4]] * 2


# ---------------------------------------------------------------- projections (Eq. 2)
@pytest.mark.parametrize("M,N,Kd", [(1, 64, 64), (127, 128, 64), (129, 256, 128), (300, 384, 192),
                                    (1024, 2304, 768), (2050, 512, 2048), (4099, 3072, 768),
                                    # CTA-pair 256x256 tiles (large M, N % 256 == 0)
                                    (8192, 2048, 512), (2600, 4608, 320), (10000, 4096, 1024)])
@pytest.mark.parametrize("act", [0, 1])
def test_linear_bf16(A, M, N, Kd, act):
    g = np.random.default_rng(M + N + Kd + act)
    x = S.round_to(g.standard_normal((M, Kd)).astype(np.float32), "bf16")
    w = S.round_to((0.05 * g.standard_normal((N, Kd))).astype(np.float32), "bf16")
    b = S.round_to((0.1 * g.standard_normal(N)).astype(np.float32), "bf16")
    out = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    A.adadsf_linear(H.to_dev(x, torch.bfloat16), H.to_dev(w, torch.bfloat16),
                    H.to_dev(b, torch.bfloat16), out, act=act)
    ref = O.linear(x, w, b, "gelu" if act else None)
    assert H.max_rel(H.to_np(out), ref) < 8e-3


@pytest.mark.parametrize("M,N,Kd,act", [(1, 64, 3072, 0), (300, 768, 3072, 1), (1384, 768, 3072, 0),
                                        (128, 256, 2048, 0), (777, 2304, 768, 1), (1000, 384, 1024, 0),
                                        (1024, 768, 768, 1), (1024, 768, 3072, 0), (333, 640, 960, 1),
                                        (129, 128, 192, 0),
                                        # fewer than 128 rows: a stage loads only them, rounded up to 8
                                        (9, 8192, 2048, 1), (17, 1024, 2048, 1), (40, 4608, 3584, 1), (100, 640, 1536, 0),
                                        # 16 rows and fewer: direct and streamed products, which never split into scratch
                                        (5, 512, 3584, 0), (13, 4608, 3584, 1), (16, 3584, 18944, 0)])
def test_linear_bf16_small_m(A, M, N, Kd, act):
    """Small-M projections of the sparse layers: one wave of tiles, long K
    (with room for scratch most of these run split along K over clusters of 2
    or 4 CTAs, with ragged M, N and K tails and uneven K ranges per CTA; with
    the minimum workspace they do not); two launches in a row agree bit for
    bit (the partial tiles are summed in a fixed order)."""
    g = np.random.default_rng(M * 7 + N + Kd)
    x = S.round_to(g.standard_normal((M, Kd)).astype(np.float32), "bf16")
    w = S.round_to((0.05 * g.standard_normal((N, Kd))).astype(np.float32), "bf16")
    b = S.round_to((0.1 * g.standard_normal(N)).astype(np.float32), "bf16")
    ref = O.linear(x, w, b, "gelu" if act else None)
    for ws_bytes in (A.LINEAR_SPLIT_WS_BYTES, 256):
        ws = A.workspace(ws_bytes)
        outs = []
        for _ in range(2):
            out = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
            A.adadsf_linear(H.to_dev(x, torch.bfloat16), H.to_dev(w, torch.bfloat16),
                            H.to_dev(b, torch.bfloat16), out, act=act, ws=ws)
            assert A.adadsf_sync_check(ws) == A.OK
            assert H.max_rel(H.to_np(out), ref) < 8e-3
            outs.append(out)
        assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("M,N,Kd", [(1, 4, 4), (65, 132, 68), (200, 2048, 512)])
def test_linear_f32(A, M, N, Kd):
    g = np.random.default_rng(M * N)
    x = g.standard_normal((M, Kd)).astype(np.float32)
    w = (0.05 * g.standard_normal((N, Kd))).astype(np.float32)
    out = torch.empty((M, N), dtype=torch.float32, device="cuda")
    A.adadsf_linear(H.to_dev(x, torch.float32), H.to_dev(w, torch.float32), None, out, act=1)
    assert H.max_rel(H.to_np(out), O.linear(x, w, None, "gelu")) < 1e-5


@pytest.mark.parametrize("M,N,Kd,act", [(1, 64, 64, 0), (7, 192, 448, 1), (8, 3072, 768, 1), (9, 2304, 768, 0),
                                        (16, 64, 3072, 0), (16, 4096, 1984, 1), (8, 1536, 8960, 0), (17, 768, 768, 0)])
def test_linear_bf16_few_rows(A, M, N, Kd, act):
    """Products of at most 16 rows: one and two 8-row halves, fewer pieces of K
    than warps and not a multiple of them, single and several tiles a block (and
    17 rows, which take the tensor-core kernels). One bf16 rounding of the output
    (2^-9 of an element, under 8e-3 of the largest)."""
    g = np.random.default_rng(M * N + Kd)
    x = S.round_to(g.standard_normal((M, Kd)).astype(np.float32), "bf16")
    w = S.round_to((g.standard_normal((N, Kd)) / np.sqrt(Kd)).astype(np.float32), "bf16")
    b = S.round_to(g.standard_normal(N).astype(np.float32), "bf16")
    out = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = A.workspace(A.LINEAR_SPLIT_WS_BYTES)
    A.adadsf_linear(*(H.to_dev(t, torch.bfloat16) for t in (x, w, b)), out[:M], act=act, ws=ws)
    assert A.adadsf_sync_check(ws) == A.OK
    ref = O.linear(x, w, b.astype(np.float64), "gelu" if act else None)
    assert H.max_rel(H.to_np(out[:M]), ref) < 8e-3
    assert bool((out[M] == 7.0).all())          # nothing past the last row


@pytest.mark.parametrize("M,N,Kd,act", [(1, 3584, 4096, 0), (8, 3584, 3968, 1), (9, 1088, 8256, 0), (16, "last", 1728, 1),
                                        (16, "past", 1728, 0), (13, 512, 16448, 0), (16, 448, 20480, 0), (1, 512, 27392, 0),
                                        (7, "last", 3136, 1)])
def test_linear_bf16_few_rows_streamed(A, M, N, Kd, act):
    """At most 16 rows and more weights than the direct kernel takes: one and two
    8-row halves, 1 to 8 groups of columns a pair of CTAs (up to 64 columns for
    each pair of SMs: the last width of that, and one past it), K of an odd number
    of 64-element blocks (and N past either end of the range, the tensor-core
    kernels). One bf16 rounding of the output (2^-9 of an element, under 8e-3 of the
    largest)."""
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    N = {"last": 64 * pairs, "past": 64 * (pairs + 1)}.get(N, N)
    g = torch.Generator(device="cuda").manual_seed(N + Kd)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    x, w, b = rnd(M, Kd).bfloat16(), (rnd(N, Kd) / Kd ** 0.5).bfloat16(), rnd(N).bfloat16()
    out = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = A.workspace(A.LINEAR_SPLIT_WS_BYTES)
    A.adadsf_linear(x, w, b, out[:M], act=act, ws=ws)
    assert A.adadsf_sync_check(ws) == A.OK
    ref = x.double() @ w.double().T + b.double()
    if act:
        ref = torch.nn.functional.gelu(ref)
    assert H.max_rel(H.to_np(out[:M]), ref.cpu().numpy()) < 8e-3
    assert bool((out[M] == 7.0).all())          # nothing past the last row
    again = torch.empty_like(out[:M])
    A.adadsf_linear(x, w, b, again, act=act, ws=ws)
    assert torch.equal(again, out[:M])


@pytest.mark.parametrize("entry", ["linear", "linear_few_rows", "router", "align_output"])
def test_first_cuda_call_of_a_host_thread(A, entry):
    """A thread's first use of CUDA is a call whose kernel loads through tensor
    maps: it is accepted and gives what the main thread gets."""
    g = torch.Generator(device="cuda").manual_seed(6)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda").bfloat16()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    if entry.startswith("linear"):
        x, w = rnd(16 if entry == "linear_few_rows" else 300, 2048), rnd(4608, 2048)
        out, ws = torch.empty(x.shape[0], 4608, dtype=torch.bfloat16, device="cuda"), A.workspace(256)
        fn, keep = A.lib().adadsf_linear, (x, w)
        args = (p(x), p(w), None, x.shape[0], 4608, 2048, A.DTYPE_CODE[x.dtype], 0, p(out), p(ws), ws.numel(), stream)
    elif entry == "router":
        shape = S.PYTHIA_160M.replace(n_layers=1)
        w, x = A.to_device(H.host_layer(shape, 3), torch.bfloat16), rnd(8192, shape.d)
        cfg, lw = A.make_cfg(shape), A.layer_struct(w)
        out, ws = torch.empty(8192, device="cuda"), A.workspace(256)
        fn, keep = A.lib().adadsf_router_scores, (x, w)
        args = (ctypes.byref(cfg), ctypes.byref(lw), p(x), 8192, p(out), p(ws), ws.numel(), stream)
    else:
        hs, hd, head = rnd(200, 512), rnd(200, 512), rnd(640, 512)
        out = torch.zeros(2, dtype=torch.float64, device="cuda")
        ws = A.workspace(A.lib().adadsf_align_workspace_size(200, 640))
        fn, keep = A.lib().adadsf_align_output, (hs, hd, head)
        args = (p(hs), p(hd), p(head), 200, 512, 640, A.DTYPE_CODE[hs.dtype], p(out), p(ws), ws.numel(), stream)
    torch.cuda.synchronize()
    assert fn(*args) == A.OK
    torch.cuda.synchronize()
    ref = out.clone()
    out.zero_()
    torch.cuda.synchronize()
    status = []
    t = threading.Thread(target=lambda: status.append(fn(*args)))
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert status == [A.OK] and torch.equal(out, ref) and len(keep)


def test_linear_from_two_host_threads(A):
    """Streamed products of different column counts (so different sizes of the
    same kernel's ring) enqueued by two host threads on streams of their own:
    none is refused, and each output is the one it gets alone. The calls go
    straight to the library, whose part of a call outside the interpreter's lock
    is then the longer one: the threads meet there."""
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda").bfloat16()
    jobs = [(rnd(16, k), rnd(n, k)) for n, k in ((4608, 2048), (512, 20480))]
    outs = [torch.empty(16, w.shape[0], dtype=torch.bfloat16, device="cuda") for _, w in jobs]
    wss, streams = [A.workspace(256) for _ in jobs], [torch.cuda.Stream() for _ in jobs]
    fn = A.lib().adadsf_linear
    vp = ctypes.c_void_p
    calls = [(vp(x.data_ptr()), vp(w.data_ptr()), None, 16, w.shape[0], w.shape[1], A.DTYPE_CODE[x.dtype], 0,
              vp(o.data_ptr()), vp(ws.data_ptr()), ws.numel(), vp(st.cuda_stream))
             for (x, w), o, ws, st in zip(jobs, outs, wss, streams)]
    torch.cuda.synchronize()
    assert [fn(*c) for c in calls] == [A.OK, A.OK]
    torch.cuda.synchronize()
    alone = [o.clone() for o in outs]
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    refused, last, start = [0, 0], [], threading.Barrier(2)

    def work(i):
        start.wait()
        for _ in range(20000):
            if fn(*calls[i]) != A.OK:
                refused[i] += 1
                last.append(A.adadsf_last_error())
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert refused == [0, 0], last
    assert all(A.adadsf_sync_check(ws) == A.OK for ws in wss)
    assert torch.equal(outs[0], alone[0]) and torch.equal(outs[1], alone[1])


@pytest.mark.parametrize("M,N,Kd,act", [(1, 4, 4, 0), (63, 36, 100, 1), (65, 516, 2052, 0), (129, 68, 64, 1),
                                        (64, 512, 2048, 0), (700, 2048, 96, 1), (1532, 512, 2048, 0), (3001, 260, 36, 1)])
def test_linear_f32_splits(A, M, N, Kd, act):
    """Rows, columns and k around the edges of both fp32 tiles (64 x 32 and
    128 x 64, 32 k a stage) and every cluster split of k. Error of an fp32 sum
    of K random products against its result: under sqrt(K) 2^-24 of its rms, and
    under 10 of that on the largest of 10^6 elements (3e-5 at K = 2052)."""
    g = np.random.default_rng(M * N + Kd)
    x = g.standard_normal((M, Kd)).astype(np.float32)
    w = (0.05 * g.standard_normal((N, Kd))).astype(np.float32)
    b = g.standard_normal(N).astype(np.float32)
    out = torch.full((M + 1, N), 7.0, device="cuda")
    A.adadsf_linear(H.to_dev(x, torch.float32), H.to_dev(w, torch.float32), H.to_dev(b, torch.float32), out[:M], act=act)
    ref = O.linear(x, w, b.astype(np.float64), "gelu" if act else None)
    H.assert_close(out[:M].cpu().numpy(), ref, 3e-5, "linear f32")
    assert bool((out[M] == 7.0).all())          # nothing past the last row


# ---------------------------------------------------------------- router (Sec. 3.4)
@pytest.mark.parametrize("n,d,h", [(1, 64, 1), (15, 512, 64), (17, 192, 65), (128, 2048, 200), (2044, 512, 64)])
def test_router_f32_edges(A, n, d, h):
    """Rows around the 16-row blocks, feature widths that leave warps idle, and
    hidden widths that are not a multiple of the 64 units of a tile. fp32 sums of
    d products, then of h: under 2e-6 of the scores' rms."""
    shape = S.PYTHIA_70M.replace(d=d, router_hidden=h, n_layers=1)
    W = H.host_layer(shape, n + h)
    x = S.hidden(n, 1, n, d)[0]
    sc = torch.full((n + 1,), 7.0, device="cuda")
    A.adadsf_router_scores(A.make_cfg(shape), A.to_device(W, torch.float32), H.to_dev(x, torch.float32), sc[:n])
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    assert H.elem_rel(sc[:n].cpu().numpy(), ref) < 1e-5
    assert float(sc[n]) == 7.0


@pytest.mark.parametrize("per_sm,off,d", [(0, 1, 64), (0, 15, 3584), (0, 17, 192), (4, 0, 1536), (4, 1, 1536),
                                          (8, -3, 768), (8, 1, 768), (16, 0, 2048), (16, 1, 2048)])
def test_router_few_tokens(A, per_sm, off, d):
    """bf16 scores around the 16-token blocks, every cluster width (8, 4 and 2 CTAs
    take up to 4, 8 and 16 tokens an SM), widths with fewer 32-feature pieces than
    CTAs, and past the last width the 128-token tiles. Products are exact; an fp32
    sum of d, then of 64 units: under 1e-5 of the scores' rms (2e-6 in rms measured
    for the tiles)."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + off
    shape = S.PYTHIA_160M.replace(d=d, n_layers=1)
    W = H.host_layer(shape, n + d)
    x = S.round_to(S.hidden(n, 1, n, d)[0], "bf16")
    outs = []
    for _ in range(2):
        sc = torch.full((n + 1,), 7.0, device="cuda")
        A.adadsf_router_scores(A.make_cfg(shape), A.to_device(W, torch.bfloat16), H.to_dev(x, torch.bfloat16), sc[:n])
        outs.append(sc.cpu())
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    assert H.elem_rel(outs[0][:n].numpy(), ref) < 1e-5
    assert float(outs[0][n]) == 7.0 and torch.equal(*outs)


@pytest.mark.parametrize("shape,n", [(S.PYTHIA_160M, 1), (S.PYTHIA_160M, 2048), (S.QWEN25_1_5B, 333),
                                     (S.PYTHIA_70M, 128), (S.PYTHIA_160M, 777), (S.PYTHIA_1_4B, 16384)])
def test_router(A, shape, n):
    W = H.host_layer(shape, 3)
    x = S.round_to(np.random.default_rng(n).standard_normal((n, shape.d)).astype(np.float32), shape.dtype)
    w = A.to_device(W, H.tdtype(shape))
    sc = torch.empty(n, dtype=torch.float32, device="cuda")
    A.adadsf_router_scores(A.make_cfg(shape), w, H.to_dev(x, H.tdtype(shape)), sc)
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    err = np.max(np.abs(sc.cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err < (5e-3 if shape.dtype == "bf16" else 1e-5)


@pytest.mark.parametrize("shape,n", [(S.PYTHIA_160M, 2048), (S.PYTHIA_160M, 2600), (S.PYTHIA_1_4B, 16384),
                                     (S.QWEN25_1_5B, 999), (S.QWEN25_1_5B, 3001),
                                     (S.QWEN25_7B.replace(ffn=256), 4096),
                                     (S.QWEN25_7B.replace(ffn=256), 25600 - 77)])
def test_router_split(A, shape, n):
    """Router with room for scratch. Up to 16 tokens an SM (2048 and 999 here)
    it is not used. Past that and up to one wave of 128-token tiles every
    CTA takes whole tiles; past it (the last case: 200 tiles of d = 3584 on
    the GPU's ~150 SMs) the CTAs take equal ranges of k-blocks, tiles are
    split along d and the last CTA of a tile sums the partials in a fixed
    order. Either way two calls agree bit for bit and the counters end at
    zero."""
    W = H.host_layer(shape, 3)
    x = S.round_to(np.random.default_rng(n + 1).standard_normal((n, shape.d)).astype(np.float32), shape.dtype)
    w = A.to_device(W, H.tdtype(shape))
    cfg = A.make_cfg(shape)
    ws = A.workspace(A.adadsf_router_select_workspace_size(cfg, 1, 1))
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    outs = []
    for _ in range(2):
        sc = torch.empty(n, dtype=torch.float32, device="cuda")
        A.adadsf_router_scores(cfg, w, H.to_dev(x, H.tdtype(shape)), sc, ws=ws)
        assert A.adadsf_sync_check(ws) == A.OK
        err = np.max(np.abs(sc.cpu().numpy() - ref)) / np.max(np.abs(ref))
        assert err < 5e-3
        outs.append(sc)
    assert torch.equal(outs[0], outs[1])
    assert int(ws[256:256 + SYNC_BYTES].view(torch.int32).abs().sum()) == 0


@pytest.mark.parametrize("shape,B,T,K", [(S.PYTHIA_70M, 2, 128, 64),
                                         (S.PYTHIA_160M, 4, 512, 256), (S.PYTHIA_1_4B, 8, 2048, 1024),
                                         (S.QWEN25_1_5B, 3, 333, 100), (S.PYTHIA_160M, 2, 100, 1),
                                         (S.PYTHIA_160M, 5, 64, 64), (S.PYTHIA_160M, 300, 1, 1),
                                         (S.QWEN25_7B.replace(ffn=256), 2, 4096, 2000), (S.PYTHIA_160M, 1, 16384, 777)])
def test_router_select(A, shape, B, T, K):
    """Router scores and the per-sequence Top-K in one launch (Sec. 3.4):
    scores within the router tolerance of the oracle, and the kept positions
    bit-exact against the oracle's Top-K of the GPU's own scores; the
    counters in the workspace end at zero, so a second call selects the same."""
    W = H.host_layer(shape, 5)
    g = np.random.default_rng(B * 1000 + T + K)
    x = S.round_to(g.standard_normal((B * T, shape.d)).astype(np.float32), shape.dtype)
    w = A.to_device(W, H.tdtype(shape))
    cfg = A.make_cfg(shape)
    ws = A.workspace(A.adadsf_router_select_workspace_size(cfg, B, T))
    ref = O.router_scores(x.astype(np.float64), H.f64(W))
    xd = H.to_dev(x, H.tdtype(shape))
    first = None
    for rep in range(2):
        sc = torch.empty(B * T, dtype=torch.float32, device="cuda")
        idx = torch.full((B, K), -1, dtype=torch.int32, device="cuda")
        rows = torch.full((B, K), -1, dtype=torch.int32, device="cuda")
        A.adadsf_router_select(cfg, w, xd, B, T, K, sc, idx, rows, ws=ws)
        assert A.adadsf_sync_check(ws) == A.OK
        s = sc.cpu().numpy()
        assert np.max(np.abs(s - ref)) / np.max(np.abs(ref)) < 5e-3
        gi, gr = idx.cpu().numpy(), rows.cpu().numpy()
        for b in range(B):
            kept = O.topk_keep(s[b * T:(b + 1) * T], K)
            assert gi[b].tolist() == kept.tolist(), b
            assert gr[b].tolist() == (b * T + kept).tolist(), b
        if first is None:
            first = (sc, idx)
        else:
            assert torch.equal(first[0], sc) and torch.equal(first[1], idx)
    assert int(ws[256:256 + SYNC_BYTES].view(torch.int32).abs().sum()) == 0


# ---------------------------------------------------------------- attention (Eq. 1)
@pytest.mark.parametrize("hq,hkv,hd", [(12, 12, 64), (12, 2, 128), (4, 4, 128)])
@pytest.mark.parametrize("B,K", [(1, 1), (2, 63), (2, 64), (3, 130), (1, 257)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_attention(A, hq, hkv, hd, B, K, dtype):
    shape = S.PYTHIA_160M.replace(n_heads=hq, n_kv_heads=hkv, head_dim=hd, d=hq * hd if hq * hd % 64 == 0 else 768,
                                  dtype=dtype)
    width = (hq + 2 * hkv) * hd
    g = np.random.default_rng(B * K + hq + hd)
    qkv = S.round_to(g.standard_normal((B * K, width)).astype(np.float32), dtype)
    out = torch.empty((B * K, hq * hd), dtype=H.tdtype(shape), device="cuda")
    A.adadsf_causal_attention(A.make_cfg(shape), H.to_dev(qkv, H.tdtype(shape)), B, K, out)
    got = H.to_np(out)
    q64 = qkv.astype(np.float64)
    for b in range(B):
        blk = q64[b * K:(b + 1) * K]
        ref = O.causal_attention(blk[:, :hq * hd], blk[:, hq * hd:(hq + hkv) * hd], blk[:, (hq + hkv) * hd:],
                                 hq, hkv, hd)
        assert H.max_rel(got[b * K:(b + 1) * K], ref) < (2e-2 if dtype == "bf16" else 1e-5)


@pytest.mark.parametrize("hq,hkv,hd,B,K", [(8, 8, 64, 1, 65), (8, 2, 64, 3, 128), (2, 1, 128, 2, 383), (1, 1, 64, 1, 700),
                                           (8, 2, 64, 1, 8), (8, 2, 64, 1, 9), (8, 2, 64, 40, 16), (8, 8, 64, 40, 17),
                                           (2, 1, 128, 3, 1), (16, 4, 128, 30, 13)])
def test_attention_f32_tiles(A, hq, hkv, hd, B, K):
    """Key and query tiles of 64 of the fp32 kernel, both sides of the lines to the
    one for short sequences (8 keys, 16 with many heads), and causality to the bit: an
    infinite value and a NaN key of the last token leave every earlier row as it
    was. fp32 softmax and sums over K keys: within 1e-5 of the largest element."""
    shape = S.PYTHIA_160M.replace(n_heads=hq, n_kv_heads=hkv, head_dim=hd, d=hq * hd, dtype="f32")
    width = (hq + 2 * hkv) * hd
    g = np.random.default_rng(B * K + hq)
    qkv = g.standard_normal((B * K, width)).astype(np.float32)
    out = torch.empty((B * K, hq * hd), device="cuda")
    A.adadsf_causal_attention(A.make_cfg(shape), H.to_dev(qkv, torch.float32), B, K, out)
    for b in range(B):
        blk = qkv[b * K:(b + 1) * K].astype(np.float64)
        ref = O.causal_attention(blk[:, :hq * hd], blk[:, hq * hd:(hq + hkv) * hd], blk[:, (hq + hkv) * hd:],
                                 hq, hkv, hd)
        assert H.max_rel(out[b * K:(b + 1) * K].cpu().numpy(), ref) < 1e-5
    qkv.reshape(B, K, width)[:, -1, (hq + hkv) * hd:] = np.inf
    qkv.reshape(B, K, width)[:, -1, hq * hd:(hq + hkv) * hd] = np.nan
    again = torch.empty_like(out)
    A.adadsf_causal_attention(A.make_cfg(shape), H.to_dev(qkv, torch.float32), B, K, again)
    assert torch.equal(again.view(B, K, -1)[:, :-1], out.view(B, K, -1)[:, :-1])


@pytest.mark.parametrize("hq,hkv,hd,B,K", [(12, 12, 64, 7, 520), (12, 12, 64, 7, 300), (12, 2, 128, 5, 520),
                                          (4, 4, 128, 20, 300), (28, 4, 128, 2, 1100)])
def test_attention_paired_tiles(A, hq, hkv, hd, B, K):
    """Enough (query-block pair, head, sequence) work units to fill the GPU:
    the kernel runs two query tiles per CTA (with an odd number of query
    blocks the last pair has one tile), bf16 against the oracle."""
    shape = S.PYTHIA_160M.replace(n_heads=hq, n_kv_heads=hkv, head_dim=hd, d=hq * hd, dtype="bf16")
    width = (hq + 2 * hkv) * hd
    g = np.random.default_rng(B * K + hq + hd + 7)
    qkv = S.round_to(g.standard_normal((B * K, width)).astype(np.float32), "bf16")
    out = torch.empty((B * K, hq * hd), dtype=torch.bfloat16, device="cuda")
    A.adadsf_causal_attention(A.make_cfg(shape), H.to_dev(qkv, torch.bfloat16), B, K, out)
    got = H.to_np(out)
    q64 = qkv.astype(np.float64)
    for b in range(B):
        blk = q64[b * K:(b + 1) * K]
        ref = O.causal_attention(blk[:, :hq * hd], blk[:, hq * hd:(hq + hkv) * hd], blk[:, (hq + hkv) * hd:],
                                 hq, hkv, hd)
        assert H.max_rel(got[b * K:(b + 1) * K], ref) < 2e-2


# ---------------------------------------------------------------- Eq. 4 statistics
@pytest.mark.parametrize("n,d,dtype", [(1, 64, "f32"), (37, 768, "bf16"), (5000, 1536, "bf16"),
                                       (3000, 512, "f32")])
def test_layer_stats(A, n, d, dtype):
    g = np.random.default_rng(n + d)
    a = S.round_to(g.standard_normal((n, d)).astype(np.float32), dtype)
    b = S.round_to((a + 0.7 * g.standard_normal((n, d))).astype(np.float32), dtype)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    ad, bd = H.to_dev(a, td), H.to_dev(b, td)
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_layer_stats(ad, bd, acc)
    A.adadsf_layer_stats(ad, ad, acc)                    # accumulates: + n rows of cos = 1
    ref, cnt = O.cos_sim_stat(a.astype(np.float64), b.astype(np.float64))
    got = acc.cpu().numpy()
    assert got[1] == 2 * n
    assert got[0] == pytest.approx(ref + n, rel=1e-5)
    flat = torch.zeros(3, dtype=torch.float64, device="cuda")
    A.adadsf_layer_stats(ad, bd, flat, mode=A.STATS_FLAT)
    assert flat.cpu().numpy() == pytest.approx(O.cos_sim_stat(a.astype(np.float64), b.astype(np.float64), "flat"),
                                               rel=1e-5)
    again = torch.zeros(2, dtype=torch.float64, device="cuda")
    A.adadsf_layer_stats(ad, bd, again)
    A.adadsf_layer_stats(ad, ad, again)
    assert again.cpu().numpy().tolist() == got.tolist()  # bit-reproducible


@pytest.mark.parametrize("n,d,dtype", [(31, 8, "bf16"), (32, 264, "bf16"), (33, 4, "f32"), (0, 2048, "bf16"), (1, 516, "f32"),
                                       (70001, 72, "bf16")])
def test_layer_stats_row_groups(A, n, d, dtype):
    """Rows summed 32 at a time: last groups short, full and of one row, as many
    groups as SMs and one more (n 0 and 1: the last that takes a warp per row, and
    the first that does not), and more groups than blocks. A row's fp32 sums hold d / 32 + 5 roundings at most, a
    cosine three such sums, so well under 1e-5 each; the sum over rows is fp64."""
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    n += 32 * torch.cuda.get_device_properties(0).multi_processor_count if n < 2 else 0
    gen = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randn((n, d), generator=gen, device="cuda").to(td)
    b = (a.float() + 0.7 * torch.randn((n, d), generator=gen, device="cuda")).to(td)
    acc = torch.zeros(2, dtype=torch.float64, device="cuda")
    flat = torch.zeros(3, dtype=torch.float64, device="cuda")
    A.adadsf_layer_stats(a, b, acc)
    A.adadsf_layer_stats(a, b, flat, mode=A.STATS_FLAT)
    a, b = a.double(), b.double()
    dot, na, nb = (a * b).sum(1), (a * a).sum(1), (b * b).sum(1)
    assert acc[1].item() == n
    assert acc[0].item() == pytest.approx((dot / (na.sqrt() * nb.sqrt())).sum().item(), rel=1e-5)
    assert flat.tolist() == pytest.approx([dot.sum().item(), na.sum().item(), nb.sum().item()], rel=1e-5)


# ---------------------------------------------------------------- weights written just before
@pytest.mark.parametrize("M,N,Kd", [(3, 768, 1024), (8, 1024, 14336), (16, 4608, 2048), (60, 1024, 2048), (300, 512, 1024),
                                    (4096, 1024, 2048)])
def test_linear_on_weights_written_just_before(A, M, N, Kd):
    """A product whose weights the call before it on the stream writes (every
    kernel that requests weights ahead of its turn: direct and streamed few-row
    products, split along K, one and two CTAs a tile): the weights are the new
    ones, to the bit what the product gives after a synchronisation."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda").bfloat16()
    x, mix = rnd(M, Kd), (rnd(Kd, 512) / 16).bfloat16()
    base = [rnd(N, 512) for _ in range(6)]
    w, out = torch.zeros(N, Kd, dtype=torch.bfloat16, device="cuda"), rnd(M, N)
    ws = A.workspace(A.LINEAR_SPLIT_WS_BYTES)
    got = []
    for b in base:
        A.adadsf_linear(b, mix, None, w, ws=ws)
        A.adadsf_linear(x, w, None, out, ws=ws)
        got.append(out.clone())
    assert A.adadsf_sync_check(ws) == A.OK
    for b, o in zip(base, got):
        A.adadsf_linear(b, mix, None, w, ws=ws)
        torch.cuda.synchronize()
        A.adadsf_linear(x, w, None, out, ws=ws)
        assert torch.equal(out, o)


@pytest.mark.parametrize("n", [100, 2000, 8192])
def test_router_on_weights_written_just_before(A, n):
    """The same for router scores whose W1 (and the rest) was just written."""
    shape = S.PYTHIA_160M.replace(n_layers=1, d=2048)
    W = [A.to_device(H.host_layer(shape, 5 + i), torch.bfloat16) for i in range(2)]
    x = H.to_dev(S.hidden(n, 1, n, shape.d)[0], torch.bfloat16)
    g = torch.Generator(device="cuda").manual_seed(n)
    mix = (torch.randn((shape.d, shape.d), generator=g, device="cuda") / 32).bfloat16()
    live = {k: v.clone() for k, v in W[0].items()}
    cfg, ws = A.make_cfg(shape), A.workspace(256)
    sc = torch.empty(n, device="cuda")

    def scores(src, wait):
        A.adadsf_linear(src["router_w1"], mix, None, live["router_w1"], ws=ws)
        if wait:
            torch.cuda.synchronize()
        A.adadsf_router_scores(cfg, live, x, sc)
        return sc.clone()
    got = [scores(W[i % 2], False) for i in range(6)]
    ref = [scores(W[i], True) for i in range(2)]
    assert all(torch.equal(s, ref[i % 2]) for i, s in enumerate(got)) and not torch.equal(*ref)


@pytest.mark.parametrize("rot", [0, 64])
def test_layer_on_weights_folded_just_before(A, rot):
    """A dense layer right behind adadsf_fold_norms of its weights; without
    rotary its norm is the first launch, which reads what the folding stores last."""
    shape = S.PYTHIA_160M.replace(n_layers=1, rotary_dim=rot)
    cfg = A.make_cfg(shape)
    x0 = H.to_dev(S.hidden(9, 2, 64, shape.d), torch.bfloat16)
    ws = A.workspace(A.adadsf_layer_workspace_size(cfg, 2, 64, 64))
    outs = []
    for wait in (False, False, True):
        W = A.to_device(H.host_layer(shape, 6), torch.bfloat16)
        x = x0.clone()
        torch.cuda.synchronize()
        A.adadsf_fold_norms(cfg, W)
        if wait:
            torch.cuda.synchronize()
        A.adadsf_sparse_layer_forward(cfg, W, x, 64, ws=ws)
        outs.append(x)
    assert A.adadsf_sync_check(ws) == A.OK
    assert torch.equal(outs[0], outs[2]) and torch.equal(outs[1], outs[2])
