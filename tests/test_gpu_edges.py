"""The kernels at the sizes where they can go wrong: edges of tiles, remainders, the
smallest and the largest of each form's range, against the fp64 oracle.

Bounds.  bf16: the two operands of a product and the output are rounded to 8 significant bits,
each by at most 2^-8 of an element and, over many, by 1.7e-3 < 2^-9 of the norm; sums are
fp32: 3 * 2^-9 in the norm (BF16).  fp32: a sum of n
terms in any order errs by about sqrt(n) * 2^-24 of its norm for these random signs: 4e-6 for
4096 terms, through the three kernels of the longest chain, and 1.1e-5 for the one sum of
32784 terms in the exact mode: F32 = 1.2e-5.  The fp32 products alone, over up to 1000 terms,
measure 1.1e-7 from split operands and 2.9e-7 on FFMA; without any one of the six products of
parts it would be 2e-6 and more: SPLIT = 6e-7.
"""
import ctypes
import threading
import time

import numpy as np
import pytest
import torch

import paper_2309_15275_b200 as lbp
from oracle import lbp_oracle as O

pytestmark = pytest.mark.gpu

BF16 = 3 * 2.0 ** -9
F32 = 1.2e-5
SPLIT = 6e-7


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def f64(t):
    return t.detach().cpu().to(torch.float64).numpy()


def rel(got, want):
    return O.rel_fro(f64(got), want)


def draw(dev, seed, *shape, dtype=torch.bfloat16, scale=1.0):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(shape, generator=g) * scale).to(dtype).to(dev)


def layer(dev, seed, B, H, W, ci, co, dtype=torch.bfloat16):
    return (draw(dev, seed, B, H, W, ci, dtype=dtype), draw(dev, seed + 1, B, H, W, co, dtype=dtype, scale=0.01),
            draw(dev, seed + 2, co, ci, dtype=dtype))


def want_lowrank(x, gy, w, k, bases):
    return O.backward_lowrank_padded(f64(x), f64(gy), f64(w), k, bases)


def tri(n):
    return [(i, j) for i in range(n) for j in range(n) if i + j < n]


# one set per form of the expansion, with rows that start at j = 0 and without
FORMS = {
    "dc": [(0, 0)],
    "2": [(0, 0), (1, 0), (0, 1)],
    "2_holes": [(1, 1), (0, 1)],
    "4": [(3, 0), (0, 0), (0, 3), (1, 2), (1, 0), (0, 1), (0, 2), (1, 1)],
    "4_holes": [(0, 2), (3, 1), (2, 3)],
    "sparse": tri(4) + [(4, 0), (0, 4), (1, 3)],
    "sparse_holes": [(0, 0), (2, 5), (6, 1)],
    "no_hh": tri(4) + [(0, 4), (0, 5), (4, 0), (5, 1)],
    "8": tri(8),
    "8_holes": [(7, 7), (0, 0), (4, 5), (2, 1)],
}


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("k,ci,co,B,H,W", [
    (8, 64, 64, 1, 8, 8),          # one block, half a channel tile
    (8, 136, 72, 3, 17, 23),       # CTA pairs, 8 channels past a tile, ragged grid
    (16, 264, 320, 5, 33, 16),     # 8 channels past a pair's tile
    (4, 72, 200, 9, 7, 9),
])
def test_products_kernel_forms(dev, form, k, ci, co, B, H, W):
    bases = FORMS[form]
    if any(max(b) >= k for b in bases):
        pytest.skip("the set needs a higher order")
    x, gy, w = layer(dev, 11, B, H, W, ci, co)
    ox, ow = want_lowrank(x, gy, w, k, bases)
    ws = lbp.alloc_workspace(x, gy, k, len(bases))
    gx, gw = lbp.lbp_backward(x, gy, w, k, bases, ws=ws)
    assert lbp.lbp_poll_status(ws) == 0
    assert rel(gx, ox) <= BF16 and rel(gw, ow) <= BF16
    # from coefficients taken earlier, accumulating, with a token outside the grid
    xe, ge = draw(dev, 5, B, ci), draw(dev, 6, B, co, scale=0.01)
    oxe, owe = O.backward_extra_tokens(f64(xe), f64(ge), f64(w))
    gw2, gxe = gw.clone(), torch.empty_like(xe)
    gx2, _ = lbp.lbp_backward_ex(None, gy, w, k, bases, x_hat=lbp.lbp_project(x, k, bases), beta=0.5,
                                 x_extra=xe, gy_extra=ge, gx_extra=gxe, g_W=gw2)
    assert rel(gx2, ox) <= BF16 and rel(gxe, oxe) <= BF16
    assert rel(gw2, ow + owe + 0.5 * f64(gw)) <= BF16


@pytest.mark.parametrize("ci,co,T", [(64, 64, 1), (8, 8, 130), (136, 264, 65), (256, 128, 128), (128, 520, 2049)])
def test_exact_mode_edges(dev, ci, co, T):
    # 16 tokens; tiles with a few rows or channels past their edge; many K slices
    x, gy, w = layer(dev, 21, 1, 4, 4 * T, ci, co)
    bases = [(i, j) for i in range(4) for j in range(4)]
    gx, gw = lbp.lbp_backward(x, gy, w, 4, bases)
    ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    assert rel(gx, ox) <= 2.0 ** -9 and rel(gw, ow) <= F32   # operands are taken as they are


@pytest.mark.parametrize("ci,co,B,H,W", [(64, 64, 1, 1, 1), (136, 264, 1, 1, 1), (72, 200, 1, 3, 5), (264, 72, 7, 3, 3),
                                         (128, 128, 1, 7, 37)])
def test_exact_mode_with_odd_token_counts(dev, ci, co, B, H, W):
    # 1, 15, 63 and 259 tokens: tiles of one row, k-blocks that end early or hold one token more
    x, gy, w = layer(dev, 23, B, H, W, ci, co)
    gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8)
    ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    # a product of two bf16 numbers is exact in fp32: of one token g_W holds nothing else; g_x is
    # rounded once, with as few elements as here to be held to the bound of each
    assert rel(gx, ox) <= 2.0 ** -8 and rel(gw, ow) <= (0.0 if B * H * W == 1 else F32)


@pytest.mark.parametrize("k,r", [(4, 1), (4, 4), (4, 5), (4, 9), (4, 15), (8, 1), (8, 16), (8, 17), (8, 33),
                                 (8, 48), (16, 1), (16, 16), (16, 31), (16, 48)])
@pytest.mark.parametrize("C,B,H,W", [(8, 1, 16, 16), (200, 3, 20, 36), (64, 70, 13, 12)])
def test_projection_edges(dev, k, r, C, B, H, W):
    # every width of the basis operand; less than a chunk of channels, a last chunk of 8,
    # strips of four blocks that end early, more items than CTAs with a ragged last one
    t = draw(dev, 31, B, H, W, C)
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    got = lbp.lbp_project(t, k, bases)
    want = O.project_padded(f64(t), k, bases)
    assert rel(got, want) <= 2.0 ** -9
    # a shift by one block or one channel leaves the norm alone, not the worst block
    d = np.sqrt(((f64(got) - want) ** 2).sum(axis=(3, 4)))
    assert np.all(d <= 2.0 ** -8 * np.sqrt((want ** 2).sum(axis=(3, 4))) + 1e-12)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("has_dc", [True, False])
@pytest.mark.parametrize("B,H,C", [(1, 4, 8), (3, 7, 264), (70, 12, 136)])
def test_bias_gradient_edges(dev, dtype, has_dc, B, H, C):
    bases = [(0, 0), (0, 1)] if has_dc else [(0, 1), (1, 0)]
    x, gy, w = layer(dev, 41, B, H, H, 64, C, dtype=dtype)
    ge, xe = draw(dev, 44, B, C, dtype=dtype), draw(dev, 45, B, 64, dtype=dtype)
    g_b = torch.full((C,), 3.0, dtype=torch.float32, device=dev)
    gw = torch.zeros((C, 64), dtype=torch.float32, device=dev)
    lbp.lbp_backward_ex(x, gy, w, 4, bases, beta=1.0, g_bias=g_b, x_extra=xe, gy_extra=ge,
                        gx_extra=torch.empty_like(xe), g_W=gw)
    want = O.bias_grad(f64(gy), f64(ge)) + 3.0
    # read from the rounded (0, 0) coefficients where they exist, else from g_y itself
    assert rel(g_b, want) <= (2.0 ** -9 if has_dc and dtype == torch.bfloat16 else F32)


@pytest.mark.parametrize("ci,co,B,H,k,r", [
    (4, 4, 1, 4, 4, 1),          # one tile of a few numbers
    (68, 132, 1, 9, 8, 3),       # four rows and columns past the 64 x 64 tiles
    (64, 64, 40, 32, 4, 3),      # g_W: one tile, hundreds of k-blocks
    (448, 1344, 1, 8, 8, 10),    # g_x: few tiles, 42 k-blocks
    (64, 192, 2, 33, 8, 64),     # exact, K no multiple of a k-block
    (256, 256, 1, 8, 8, 63),
])
def test_fp32_products_edges(dev, ci, co, B, H, k, r):
    x, gy, w = layer(dev, 51, B, H, H, ci, co, dtype=torch.float32)
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    gx, gw = lbp.lbp_backward(x, gy, w, k, bases)
    if r == k * k:
        ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    else:
        ox, ow = want_lowrank(x, gy, w, k, bases)
    assert rel(gx, ox) <= F32 and rel(gw, ow) <= F32


@pytest.mark.parametrize("co,ci,T,gw_dtype", [(64, 64, 512, torch.float32), (8, 8, 8192, torch.bfloat16),
                                              (136, 264, 4096, torch.float32), (512, 512, 4096, torch.bfloat16)])
def test_sum_of_k_slices(dev, co, ci, T, gw_dtype):
    # few g_W tiles over many rows: from 2 to well over 16 planes, and onto a g_W
    x, gy, w = layer(dev, 61, T // 64, 8, 8, ci, co)
    bases = lbp.lbp_select_bases(8, lbp.SEL_PREFIX, 21)
    _, ow = want_lowrank(x, gy, w, 8, bases)
    for beta in (0.0, 1.0):
        gw = torch.ones((co, ci), dtype=gw_dtype, device=dev)
        lbp.lbp_backward_ex(x, gy, w, 8, bases, beta=beta, g_W=gw)
        assert rel(gw, ow + beta) <= BF16


@pytest.mark.parametrize("r", [16, 17, 48])
def test_batch_equals_single_calls_at_high_rank(dev, r):
    shapes = [(768, 2304), (768, 768), (2304, 768)]
    bases = lbp.lbp_select_bases(8, lbp.SEL_PREFIX, r)
    ins = [layer(dev, 71 + 3 * i, 8, 16, 16, ci, co) for i, (ci, co) in enumerate(shapes)]
    xs, gys, ws_ = (list(v) for v in zip(*ins))
    g_xs = [torch.empty_like(x) for x in xs]
    g_Ws = [torch.empty(w.shape, dtype=torch.float32, device=dev) for w in ws_]
    wss = [lbp.alloc_workspace(x, gy, 8, r) for x, gy in zip(xs, gys)]
    for _ in range(2):
        lbp.lbp_backward_batch(xs, gys, ws_, 8, bases, g_xs=g_xs, g_Ws=g_Ws, wss=wss)
    for x, gy, w, gx, gw in zip(xs, gys, ws_, g_xs, g_Ws):
        ox, ow = want_lowrank(x, gy, w, 8, bases)
        assert rel(gx, ox) <= BF16 and rel(gw, ow) <= BF16
        # g_x has one order of summation whatever the tile plan; the K slices of g_W may differ
        gx1, gw1 = lbp.lbp_backward(x, gy, w, 8, bases)
        assert torch.equal(gx, gx1) and rel(gw, f64(gw1)) <= F32


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n_cls,bias", [(0, True), (1, True), (1, False)])
def test_module_step_through_the_extension(dev, dtype, n_cls, bias):
    # forward, backward and the bias gradient in the layer's dtype against the oracle
    ci, co, B, H = 72, 136, 3, 12
    bases = lbp.lbp_select_bases(4, lbp.SEL_L1, 2)
    lin = lbp.LbpLinear(ci, co, 4, bases, bias=bias, device=dev, dtype=dtype, grid=(H, H) if n_cls else None)
    if bias:
        lin.bias.data.copy_(draw(dev, 83, co, dtype=dtype))
    shape = (B, H, H) if n_cls == 0 else (B, n_cls + H * H)
    x = draw(dev, 81, *shape, ci, dtype=dtype).requires_grad_()
    gy = draw(dev, 82, *shape, co, dtype=dtype, scale=0.01)
    y = lin(x)
    y.backward(gy)
    w = f64(lin.weight)
    want_y = f64(x) @ w.T + (f64(lin.bias) if bias else 0.0)
    grid = (lambda t: t) if n_cls == 0 else (lambda t: t[:, n_cls:].reshape(B, H, H, -1))
    ox, ow = O.backward_lowrank_padded(grid(f64(x)), grid(f64(gy)), w, 4, bases)
    if n_cls:
        oxe, owe = O.backward_extra_tokens(f64(x)[:, :n_cls].reshape(-1, ci), f64(gy)[:, :n_cls].reshape(-1, co), w)
        ow = ow + owe
        assert rel(x.grad[:, :n_cls].reshape(-1, ci), oxe) <= (F32 if dtype == torch.float32 else BF16)
    tol = F32 if dtype == torch.float32 else BF16
    assert rel(y, want_y) <= tol and rel(grid(x.grad), ox) <= tol and rel(lin.weight.grad, ow) <= tol
    if bias:
        assert lin.bias.grad.dtype == dtype
        assert rel(lin.bias.grad, O.bias_grad(f64(gy).reshape(-1, 1, 1, co))) <= tol


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("k,r", [(4, 1), (4, 3), (4, 4), (4, 5), (4, 8), (4, 9), (4, 15), (8, 10), (8, 36), (16, 21)])
def test_infinities_stay_in_their_block_and_channel(dev, dtype, k, r):
    # a block's coefficients and its part of g_x are functions of that block alone: a token
    # that is not finite changes nothing elsewhere, bit for bit
    B, H, W, ci, co = 2, 3 * k, 6 * k + 1, 72, 136
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    x, gy, w = layer(dev, 91, B, H, W, ci, co, dtype=dtype)
    bad = gy.clone()
    at = [(0, 1, k, 5, np.inf), (0, H - 1, 4 * k + 1, 70, np.nan), (1, k, 0, 135, -np.inf), (1, 0, W - 1, 64, np.inf)]
    clean_blocks = torch.ones((B, H // k, -(-W // k)), dtype=torch.bool)
    for b, h, v, c, val in at:
        bad[b, h, v, c] = val
        clean_blocks[b, h // k, v // k] = False
    want, got = lbp.lbp_project(gy, k, bases), lbp.lbp_project(bad, k, bases)
    keep = clean_blocks[..., None, None].expand(want.shape).clone()
    for b, h, v, c, _ in at:
        keep[b, h // k, v // k] = True
    for b, h, v, c, _ in at:
        keep[b, h // k, v // k, :, c] = False
    keep = keep.to(dev)
    assert torch.equal(got[keep], want[keep]) and not torch.isfinite(got[~keep]).any()
    g_x, _ = lbp.lbp_backward(x, gy, w, k, bases)
    g_x_bad, _ = lbp.lbp_backward(x, bad, w, k, bases)
    tokens = clean_blocks.repeat_interleave(k, 1).repeat_interleave(k, 2)[:, :, :W].to(dev)
    assert torch.equal(g_x_bad[tokens], g_x[tokens])


def test_module_step_under_autocast(dev):
    # the product runs in bf16, the sum with the fp32 bias in fp32: y and the backward pass are fp32
    ci, co, B, H = 64, 96, 2, 8
    bases = lbp.lbp_select_bases(4, lbp.SEL_L1, 2)
    lin = lbp.LbpLinear(ci, co, 4, bases, bias=True, device=dev)
    x = draw(dev, 101, B, H, H, ci, dtype=torch.float32).requires_grad_()
    gy = draw(dev, 102, B, H, H, co, dtype=torch.float32, scale=0.01)
    with torch.autocast("cuda", dtype=torch.bfloat16):
        y = lin(x)
    assert y.dtype == torch.float32
    y.backward(gy)
    ox, ow = want_lowrank(x, gy, lin.weight, 4, bases)
    assert rel(x.grad, ox) <= F32 and rel(lin.weight.grad, ow) <= F32
    assert rel(lin.bias.grad, O.bias_grad(f64(gy))) <= F32


def batch_of(dev, seed, shapes, B=8, r=8):
    ins = [layer(dev, seed + 3 * i, B, 16, 16, ci, co) for i, (ci, co) in enumerate(shapes)]
    xs, gys, ws_ = (list(v) for v in zip(*ins))
    return dict(xs=xs, g_ys=gys, Ws=ws_, k=8, bases=lbp.lbp_select_bases(8, lbp.SEL_PREFIX, r),
                g_xs=[torch.empty_like(x) for x in xs],
                g_Ws=[torch.empty(w.shape, dtype=torch.float32, device=dev) for w in ws_],
                wss=[lbp.alloc_workspace(x, gy, 8, r) for x, gy in zip(xs, gys)])


def test_batch_call_waits_for_the_section_of_the_side_stream(dev):
    a = batch_of(dev, 111, [(768, 768), (256, 1024)])
    events = [None, None]
    lbp.lbp_backward_batch(**a, done_events=events)
    torch.cuda.synchronize()
    usleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p)
    held = threading.Thread(target=lambda: lbp.binding._lib().lbp_test_side_section(dev.index, usleep, 400000))
    held.start()
    time.sleep(0.1)
    t0 = time.perf_counter()
    lbp.lbp_backward_batch(**a, done_events=events)
    waited = time.perf_counter() - t0
    held.join()
    assert 0.1 < waited < 5.0


def test_batch_calls_of_two_threads_on_two_streams(dev):
    # every call's projections follow its own inputs, its products its own projections
    sets = [batch_of(dev, 131, [(768, 768), (256, 1024), (1024, 256)]), batch_of(dev, 151, [(384, 1536), (768, 384)])]
    want = []
    for s in sets:
        lbp.lbp_backward_batch(**s)
        torch.cuda.synchronize()
        want.append([t.clone() for t in s["g_xs"] + s["g_Ws"]])
    clean = [[t.clone() for t in s["xs"] + s["g_ys"]] for s in sets]
    failed = []

    def work(s, src, want):
        torch.cuda.set_device(dev)
        stream = torch.cuda.Stream(device=dev)
        with torch.cuda.stream(stream):
            for _ in range(40):
                for t in s["xs"] + s["g_ys"]:
                    t.zero_()
                for t, c in zip(s["xs"] + s["g_ys"], src):
                    t.copy_(c)
                lbp.lbp_backward_batch(**s, done_events=[None] * len(s["xs"]))
                got = s["g_xs"] + s["g_Ws"]
                if not all(torch.equal(g, w) for g, w in zip(got, want)):
                    failed.append(1)
    threads = [threading.Thread(target=work, args=v) for v in zip(sets, clean, want)]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed


def test_batch_call_beside_the_capture_of_another(dev):
    # the library's stream stays in a capture it has joined until that ends: a call on a
    # stream outside it runs on its own stream alone, and leaves the capture intact
    a = batch_of(dev, 171, [(768, 768), (256, 1024)])
    b = batch_of(dev, 181, [(384, 1536), (768, 384)])
    want = []
    for s in (a, b):
        lbp.lbp_backward_batch(**s)
        want.append([t.clone() for t in s["g_xs"] + s["g_Ws"]])
    for t in a["g_xs"] + a["g_Ws"] + b["g_xs"] + b["g_Ws"]:
        t.zero_()
    torch.cuda.synchronize()
    graph, inner, outer = torch.cuda.CUDAGraph(), torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
    with torch.cuda.stream(inner):
        graph.capture_begin(capture_error_mode="thread_local")
        lbp.lbp_backward_batch(**a)
        with torch.cuda.stream(outer):
            lbp.lbp_backward_batch(**b)
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    for s, w in zip((a, b), want):
        n = len(s["g_xs"])
        assert all(torch.equal(g, v) for g, v in zip(s["g_xs"], w[:n]))
        # other K slices of g_W on one stream: fp32 sums in another order
        assert all(rel(g, f64(v)) <= F32 for g, v in zip(s["g_Ws"], w[n:]))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_each_call_asks_for_the_workspace_it_needs(dev, dtype):
    # r = k*k: a call on x runs in the room of Eq. 2, one on x_hat wants that of its coefficients;
    # fp32: with no room for K slices at all as well
    B, H, ci, co, k = 4, 16, 64, 96, 4
    x, gy, w = layer(dev, 191, B, H, H, ci, co, dtype=dtype)
    bases = lbp.lbp_select_bases(k, lbp.SEL_LINF, k)
    code = lbp.LBP_BF16 if dtype == torch.bfloat16 else lbp.LBP_F32
    size = lambda form, **kw: lbp.lbp_workspace_bytes_ex(B, H, H, ci, co, k, code, lbp.LBP_F32, k * k,  # noqa: E731
                                                         bias=True, x_hat=form)
    ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    for n in [size(False)] + ([256 + 2 * 4 * ci * co + 4096] if dtype == torch.float32 else []):
        ws, g_b = torch.empty(n, dtype=torch.uint8, device=dev), torch.empty(co, device=dev)
        gx, gw = lbp.lbp_backward_ex(x, gy, w, k, bases, g_bias=g_b, ws=ws)
        assert rel(gx, ox) <= BF16 and rel(gw, ow) <= F32 and rel(g_b, O.bias_grad(f64(gy))) <= F32
        with pytest.raises(lbp.LbpError) as err:
            lbp.lbp_backward_ex(None, gy, w, k, bases, x_hat=lbp.lbp_project(x, k, bases), g_bias=g_b, ws=ws)
        assert err.value.status == 7
    ws = torch.empty(size(True), dtype=torch.uint8, device=dev)
    gx, gw = lbp.lbp_backward_ex(None, gy, w, k, bases, x_hat=lbp.lbp_project(x, k, bases), g_bias=g_b, ws=ws)
    assert rel(gx, ox) <= BF16 and rel(gw, ow) <= BF16


def test_other_threads_run_during_a_call(dev):
    # a call that waits (here for the section of the side stream) does not hold the interpreter
    a = batch_of(dev, 201, [(768, 768), (256, 1024)])
    lbp.lbp_backward_batch(**a)
    torch.cuda.synchronize()
    usleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p)
    held = threading.Thread(target=lambda: lbp.binding._lib().lbp_test_side_section(dev.index, usleep, 500000))
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.005)
    ticker = threading.Thread(target=tick)
    held.start(), ticker.start()
    time.sleep(0.1)
    t0 = time.perf_counter()
    lbp.lbp_backward_batch(**a)
    t1 = time.perf_counter()
    stop.set()
    held.join(), ticker.join()
    assert t1 - t0 > 0.1
    assert sum(t0 < t < t1 - 0.05 for t in ticks) >= 5


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,H,W,C,ci", [(1, 63, 65, 8, 8), (3, 64, 64, 72, 64), (5, 61, 67, 200, 16), (2, 128, 128, 1544, 8)])
def test_bias_gradient_over_many_tokens(dev, dtype, B, H, W, C, ci):
    # g_y itself is summed, by one cluster of CTAs, by several, by as many as the scratch has rows for
    x, gy, w = layer(dev, 211, B, H, W, ci, C, dtype=dtype)
    gy += 0.01     # sums that do not cancel: every row counts
    ge, xe = draw(dev, 214, B, C, dtype=dtype), draw(dev, 215, B, ci, dtype=dtype)
    for beta in (0.0, 0.5):
        g_b = torch.full((C,), 3.0, dtype=torch.float32, device=dev)
        gw = torch.zeros((C, ci), dtype=torch.float32, device=dev)
        lbp.lbp_backward_ex(x, gy, w, 4, [(0, 1)], beta=beta, g_bias=g_b, x_extra=xe, gy_extra=ge,
                            gx_extra=torch.empty_like(xe), g_W=gw)
        # fp64 sums, one rounding to fp32
        assert rel(g_b, O.bias_grad(f64(gy), f64(ge)) + 3.0 * beta) <= 2.0 ** -23


@pytest.fixture
def fp32_form(request, monkeypatch):
    monkeypatch.setenv("LBP_FP32_FORM", str(request.param))
    lbp.lbp_test_reload_env()
    yield request.param
    monkeypatch.undo()
    lbp.lbp_test_reload_env()


@pytest.mark.parametrize("fp32_form", [0, 1, 2], indirect=True)
@pytest.mark.parametrize("ci,co,T", [(4, 4, 1), (132, 68, 65), (64, 260, 1000), (320, 128, 256), (128, 1028, 60)])
def test_fp32_product_forms(dev, fp32_form, ci, co, T):
    # tiles and k-blocks of every form with 4 lanes, columns or k's past an edge, one or two
    # k-blocks an item.  Exact mode: D of either product is the result itself
    x, gy, w = layer(dev, 81, 1, 1, T, ci, co, dtype=torch.float32)
    for scale in (1.0, 2.0 ** -100, 2.0 ** 120):   # the parts down to subnormal, the sums up to 2^124
        gys = gy * scale
        gx, gw = lbp.lbp_backward_fullrank(x, gys, w, 8)
        ox, ow = O.backward_exact(f64(x), f64(gys), f64(w))
        assert rel(gx, ox) <= SPLIT and rel(gw, ow) <= SPLIT


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("per,gx_items,gw_items", [(5, (5, 2), (4, 3)), (6, (5, 2), (6, 2)), (11, (10, 1), (11, 1))])
def test_fp32_products_over_many_k_blocks(dev, monkeypatch, form, per, gx_items, gw_items):
    # odd and even numbers of k-blocks an item, the last of them ragged, a shorter last slice:
    # every stage and accumulator in use several times over
    monkeypatch.setenv("LBP_FP32_FORM", f"{form},{per}")
    lbp.lbp_test_reload_env()
    try:
        x, gy, w = layer(dev, 85, 1, 1, 645, 136, 580, dtype=torch.float32)
        plan = lbp.lbp_test_float_plan(136, 580, 645)
        assert plan["form"] == form
        assert (plan["gx_kb"], plan["gx_items"]) == gx_items and (plan["gw_kb"], plan["gw_items"]) == gw_items
        ws = lbp.alloc_workspace(x, gy, 8, 64)
        gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8, ws=ws)
        assert lbp.lbp_poll_status(ws) == 0
        ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
        assert rel(gx, ox) <= SPLIT and rel(gw, ow) <= SPLIT
    finally:
        monkeypatch.undo()
        lbp.lbp_test_reload_env()


@pytest.mark.parametrize("fp32_form", ["1", "2", "1,4", "2,4"], indirect=True)
def test_fp32_infinities_as_term_by_term(dev, fp32_form):
    # infinities and NaN reach the sums they belong to and no others; numbers whose bf16
    # neighbour is infinite stay finite
    x, gy, w = layer(dev, 91, 1, 1, 200, 136, 200, dtype=torch.float32)
    x[0, 0, 3, 5] = float("inf")
    gy[0, 0, 150, 131] = float("nan")
    w[7, 130] = -float("inf")
    gy[0, 0, 70, :] = 0.0
    x[0, 0, 70, 9] = 3.4e38
    gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8)
    X, G, Wd = x.reshape(-1, 136).double(), gy.reshape(-1, 200).double(), w.double()
    for got, want in ((gx.reshape(-1, 136).double(), G @ Wd), (gw.double(), G.t() @ X)):
        fin = torch.isfinite(want)
        assert torch.equal(torch.isfinite(got), fin) and torch.equal(torch.isnan(got), torch.isnan(want))
        assert torch.equal(got[~fin & ~torch.isnan(want)], want[~fin & ~torch.isnan(want)])
        assert ((got - want)[fin].norm() / want[fin].norm()).item() <= SPLIT


@pytest.mark.parametrize("fp32_form", [1, 2], indirect=True)
@pytest.mark.parametrize("ci,co,T", [(136, 200, 200), (448, 320, 645)])
def test_fp32_nan_leaves_the_other_sums_alone(dev, fp32_form, ci, co, T):
    x, gy, w = layer(dev, 95, 1, 1, T, ci, co, dtype=torch.float32)
    gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8)
    g2 = gy.clone()
    g2[0, 0, T - 3, 131] = float("nan")
    hx, hw = lbp.lbp_backward_fullrank(x, g2, w, 8)
    rows = [t for t in range(T) if t != T - 3]
    cols = [c for c in range(co) if c != 131]
    assert torch.equal(hx[0, 0, rows], gx[0, 0, rows]) and torch.isnan(hx[0, 0, T - 3]).all()
    assert torch.equal(hw[cols], gw[cols]) and torch.isnan(hw[131]).all()


def test_fp32_nan_costs_a_few_times_ffma_at_most(dev, monkeypatch):
    # a call whose g_y holds a NaN, or nothing else, against the FFMA kernel, whose time no value changes
    x, gy, w = layer(dev, 97, 1, 1, 640, 448, 1792, dtype=torch.float32)
    one, every = gy.clone(), torch.full_like(gy, float("nan"))
    one[0, 0, 320, 7] = float("nan")

    def us(form, g):
        monkeypatch.setenv("LBP_FP32_FORM", str(form))
        lbp.lbp_test_reload_env()
        ws = lbp.alloc_workspace(x, gy, 8, 64)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                lbp.lbp_backward_fullrank(x, g, w, 8, ws=ws)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 250)
        return best
    try:
        ffma = us(0, gy)
        for form in (1, 2):
            for g in (one, every):
                # measured: 1.3 to 2.7 of it (with a serial sum per thread 6.6 to 19)
                assert us(form, g) <= 4 * ffma
    finally:
        monkeypatch.undo()
        lbp.lbp_test_reload_env()


@pytest.mark.parametrize("ci,co,T", [(264, 136, 1), (136, 4, 200), (128, 260, 2), (64, 64, 3), (320, 128, 4), (132, 516, 5)])
def test_fp32_products_of_few_terms_round_once_a_term(dev, monkeypatch, ci, co, T):
    # sums of one to five terms: the same numbers from every form, of one term the rounded product
    x, gy, w = layer(dev, 99, 1, 1, T, ci, co, dtype=torch.float32)
    got = []
    try:
        for form in range(3):
            monkeypatch.setenv("LBP_FP32_FORM", str(form))
            lbp.lbp_test_reload_env()
            got.append(lbp.lbp_backward_fullrank(x, gy, w, 8))
    finally:
        monkeypatch.undo()
        lbp.lbp_test_reload_env()
    for gx, gw in got[1:]:
        if T <= 5:
            assert torch.equal(gw, got[0][1])
        if co <= 5:
            assert torch.equal(gx, got[0][0])
    if T == 1:
        assert torch.equal(got[1][1], gy.reshape(-1, 1) * x.reshape(1, -1))


@pytest.mark.parametrize("fp32_form", [0, 1, 2], indirect=True)
@pytest.mark.parametrize("exponent", [-104, -112, -118, -122, -124])
def test_fp32_products_of_small_numbers(dev, fp32_form, exponent):
    # g_y down to the smallest normal numbers: 320 and 256 terms of random signs err by
    # sqrt(320) * 2^-24 at most in any order, wherever in the range they lie (x and W times 64, so
    # that sums and most products of parts are normal; below 2^-120 a step of 2^-149 beside it)
    x, gy, w = layer(dev, 103, 1, 1, 320, 256, 256, dtype=torch.float32)
    x, w = x * 64, w * 64
    gy = gy * 100 * 2.0 ** exponent
    gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8)
    ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    bound = 320 ** 0.5 * 2.0 ** -24 + (2.0 ** -149 / 2.0 ** exponent if exponent < -120 else 0)
    assert rel(gx, ox) <= bound and rel(gw, ow) <= bound


@pytest.mark.parametrize("exponent", [-124, -130, -134])
def test_fp32_sums_below_the_normal_numbers(dev, monkeypatch, exponent):
    # sums around 2^(exponent + 4): whatever the form, as near as FMAs come, which round at 2^-149
    # (the tensor core cuts there)
    x, gy, w = layer(dev, 107, 1, 1, 320, 256, 256, dtype=torch.float32)
    gy = gy * 100 * 2.0 ** exponent
    ox, ow = O.backward_exact(f64(x), f64(gy), f64(w))
    err = []
    try:
        for form in range(3):
            monkeypatch.setenv("LBP_FP32_FORM", str(form))
            lbp.lbp_test_reload_env()
            gx, gw = lbp.lbp_backward_fullrank(x, gy, w, 8)
            err.append((rel(gx, ox), rel(gw, ow)))
    finally:
        monkeypatch.undo()
        lbp.lbp_test_reload_env()
    for ex, ew in err[1:]:
        assert ex <= 1.1 * err[0][0] and ew <= 1.1 * err[0][1]
