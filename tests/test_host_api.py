"""CPU-side checks of the C ABI: the library loads, exports every declared
symbol, and its host-only functions agree with the oracle bit for bit."""
import ctypes
import os
import re

import numpy as np
import pytest

import paper_2309_15275_b200 as lbp
from oracle import lbp_oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2309_15275_b200.build import build_library
    build_library()


def test_library_exports_every_declared_symbol():
    inc = os.path.join(ROOT, "include")
    header = "".join(open(os.path.join(inc, f)).read() for f in sorted(os.listdir(inc)) if f.endswith(".h"))
    declared = set(re.findall(r"^(?:int|size_t|double|long long|const char\*)\s+(lbp_[a-z_]+)\s*\(", header, re.M))
    assert declared == set(lbp.EXPORTED)
    lib = ctypes.CDLL(lbp.LIB_PATH)
    for name in declared:
        assert hasattr(lib, name), name


@pytest.mark.parametrize("k", (4, 8, 16))
def test_select_bases_bit_exact_vs_oracle(k):
    for m in range(1, 2 * k):
        assert lbp.lbp_select_bases(k, lbp.SEL_L1, m) == O.select_bases(k, O.RULE_L1, m)
    for m in range(1, k + 1):
        assert lbp.lbp_select_bases(k, lbp.SEL_LINF, m) == O.select_bases(k, O.RULE_LINF, m)
    for r in range(1, k * k + 1):
        assert lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r) == O.select_bases(k, O.RULE_PREFIX, r)


@pytest.mark.parametrize("k", (4, 8, 16))
def test_basis_matrix_bit_exact_vs_oracle(k):
    rng = np.random.default_rng(k)
    for r in (1, 3, k, k * k):
        pairs = [(int(p) // k, int(p) % k) for p in rng.permutation(k * k)[:r]]
        assert np.array_equal(lbp.lbp_basis_matrix(k, pairs), O.basis_matrix(k, pairs))


def test_flops_match_table1():
    f = O.flops(3072, 768, 49, 8)
    assert lbp.lbp_flops(3072, 768, 49, 8, 0) == f["vanilla"]
    assert lbp.lbp_flops(3072, 768, 49, 8, 1) == f["projection"]
    assert lbp.lbp_flops(3072, 768, 49, 8, 2) == f["lowrank_mm"]
    assert lbp.lbp_flops(3072, 768, 49, 8, 3) == f["reverse_projection"]
    assert lbp.lbp_flops(3072, 768, 49, 8, 4) == f["projection"] + f["lowrank_mm"] + f["reverse_projection"]
    assert lbp.lbp_flops(1, 1, 1, 1, 9) < 0


def test_argument_errors():
    with pytest.raises(lbp.LbpError) as e:
        lbp.lbp_select_bases(5, lbp.SEL_L1, 2)
    assert e.value.status == 3
    with pytest.raises(lbp.LbpError) as e:
        lbp.lbp_select_bases(8, lbp.SEL_PREFIX, 65)
    assert e.value.status == 4
    with pytest.raises(lbp.LbpError) as e:
        lbp.lbp_basis_matrix(8, [(0, 0), (0, 0)])
    assert e.value.status == 4
    with pytest.raises(lbp.LbpError) as e:
        lbp.lbp_basis_matrix(8, [(0, 8)])
    assert e.value.status == 4
    assert "basis" in lbp.lbp_status_string(4)


def test_workspace_bytes():
    n8 = lbp.lbp_workspace_bytes(128, 16, 16, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 8)
    n16 = lbp.lbp_workspace_bytes(128, 16, 16, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 16)
    rows = 512 * 8
    assert n8 >= rows * (768 + 3072) * 2 + rows * 768 * 4
    assert n16 > n8
    # a grid side that is no multiple of k is extended with zero tokens: as many blocks as 16 x 16
    assert (lbp.lbp_workspace_bytes(128, 16, 12, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 8)
            == lbp.lbp_workspace_bytes(128, 16, 16, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 8))
    assert lbp.lbp_workspace_bytes(128, 16, 0, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 8) == 0
    assert lbp.lbp_workspace_bytes(128, 16, 16, 768, 3072, 8, lbp.LBP_F32, lbp.LBP_BF16, 8) == 0   # dtype combo
    assert lbp.lbp_workspace_bytes(128, 16, 16, 768, 3072, 8, lbp.LBP_BF16, lbp.LBP_F32, 65) == 0


def test_device_calls_fail_loudly_without_cuda_tensors():
    import torch
    t = torch.zeros((1, 8, 8, 8), dtype=torch.float32)
    with pytest.raises(ValueError):
        lbp.lbp_project(t, 8, [(0, 0)], out=torch.zeros((1, 1, 1, 1, 8)), ws=torch.zeros(256, dtype=torch.uint8))


@pytest.mark.parametrize("k", (4, 8, 16))
def test_select_lhe_bit_exact_vs_oracle(k):
    rng = np.random.default_rng(40 + k)
    # distinct energies, then a quantised array with many ties
    for energy in (rng.random((k, k)), np.round(rng.random((k, k)) * 4) / 4):
        for r in (1, 2, k, k * k // 2, k * k):
            assert lbp.lbp_select_lhe(energy, k, r) == O.select_lhe(energy, k, r)


def test_select_lhe_argument_errors():
    e = np.ones((8, 8))
    for bad_r in (0, 65):
        with pytest.raises(lbp.LbpError) as err:
            lbp.lbp_select_lhe(e, 8, bad_r)
        assert err.value.status == 4
    bad = e.copy()
    bad[1, 1] = -1.0
    with pytest.raises(lbp.LbpError) as err:
        lbp.lbp_select_lhe(bad, 8, 3)
    assert err.value.status == 4
    bad[1, 1] = float("nan")
    with pytest.raises(lbp.LbpError) as err:
        lbp.lbp_select_lhe(bad, 8, 3)
    assert err.value.status == 4
    with pytest.raises(lbp.LbpError) as err:
        lbp.lbp_select_lhe(np.ones((5, 5)), 5, 3)
    assert err.value.status == 3
    assert lbp.lbp_spectrum_workspace_bytes(2, 16, 16, 64, 8, lbp.LBP_BF16) >= 2 * 16 * 16 * 64 * 2
    assert (lbp.lbp_spectrum_workspace_bytes(2, 15, 16, 64, 8, lbp.LBP_BF16)
            == lbp.lbp_spectrum_workspace_bytes(2, 16, 16, 64, 8, lbp.LBP_BF16))
    assert lbp.lbp_spectrum_workspace_bytes(2, 15, 16, 60, 8, lbp.LBP_BF16) == 0


def test_batch_arguments_are_checked_on_the_host_before_any_device_call():
    # fake (never dereferenced) device addresses: every check below happens on the
    # host, before the library touches the CUDA runtime
    from paper_2309_15275_b200 import binding as b
    lib = b._lib()
    n, k, r = 2, 8, 8
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    lays = (b.Layer * n)(b._layer(2, 16, 16, 64, 128, k, lbp.LBP_BF16, lbp.LBP_F32),
                         b._layer(2, 16, 16, 128, 64, k, lbp.LBP_BF16, lbp.LBP_F32))
    need = [lbp.lbp_workspace_bytes(2, 16, 16, 64, 128, k, lbp.LBP_BF16, lbp.LBP_F32, r),
            lbp.lbp_workspace_bytes(2, 16, 16, 128, 64, k, lbp.LBP_BF16, lbp.LBP_F32, r)]
    MB = 1 << 20
    base = 1 << 32

    def arr(vals):
        return (ctypes.c_void_p * n)(*vals)

    def call(x, gy, w, gx, gw, ws, sizes=None):
        sz = (ctypes.c_size_t * n)(*(sizes or need))
        return lib.lbp_backward_batch(n, arr(x), arr(gy), arr(w), arr(gx), arr(gw), lays,
                                      b._bases(bases), r, arr(ws), sz, None, None)

    x = [base, base + 64 * MB]
    gy = [base + 8 * MB, base + 72 * MB]
    w = [base + 16 * MB, base + 80 * MB]
    gx = [base + 24 * MB, base + 88 * MB]
    gw = [base + 32 * MB, base + 96 * MB]
    ws = [base + 40 * MB, base + 104 * MB]
    # g_x of problem 0 is x of problem 1
    assert call([x[0], gx[0]], gy, w, gx, gw, ws) == 12
    # the two problems share an output
    assert call(x, gy, w, gx, [gw[0], gw[0]], ws) == 12
    # workspace of problem 1 overlaps g_y of problem 0
    assert call(x, gy, w, gx, gw, [ws[0], gy[0]]) == 12
    # shared inputs are allowed: the next check that fails is the workspace size
    assert call([x[0], x[0] + 0], gy, [w[0], w[0]], gx, gw, ws, sizes=[need[0], 16]) in (2, 7)
    assert call(x, gy, w, gx, gw, ws, sizes=[need[0], need[1] - 1]) == 7
    assert call(x, gy, w, [gx[0], gx[1] + 2], gw, ws) == 6          # misaligned pointer
    assert call(x, gy, w, [gx[0], None], gw, ws) == 1               # null pointer
    assert lib.lbp_backward_batch(0, arr(x), arr(gy), arr(w), arr(gx), arr(gw), lays,
                                  b._bases(bases), r, arr(ws), (ctypes.c_size_t * n)(*need), None, None) == 2
    assert "overlap" in lbp.lbp_status_string(12)


@pytest.mark.parametrize("Cin,Cout,G,bpt,units,pair", [
    (768, 2304, 32, 16, 74, 1), (768, 768, 32, 16, 74, 1), (768, 3072, 32, 16, 74, 1),
    (3072, 768, 32, 16, 74, 1), (1024, 4096, 25, 21, 74, 1), (48, 192, 196, 16, 148, 0),
    (192, 48, 196, 16, 148, 0), (64, 64, 1, 4, 148, 0), (768, 3072, 5, 2, 66, 1)])
def test_tile_plan_covers_every_tile_once(Cin, Cout, G, bpt, units, pair):
    # what the products kernel is told to do: every tile of both products exactly
    # once, GX tiles (long epilogue) ahead of GW tiles on every unit
    max_splits = 8
    info, lists = lbp.lbp_test_tile_plan(Cin, Cout, G, bpt, 8, units, pair, max_splits)
    row_tile = 256 if pair else 128
    step = 128 if pair else 64
    assert info["BNw"] % step == 0 and info["BNx"] % step == 0 and info["BNw"] <= 256 and info["BNx"] <= 256
    assert 1 <= info["splits"] <= max_splits
    assert info["kbps"] * info["splits"] >= 2 * G > info["kbps"] * (info["splits"] - 1)
    n_gw = -(-Cout // row_tile) * -(-Cin // info["BNw"]) * info["splits"]
    n_gx = (-(-G // 2) if pair else G) * -(-Cin // info["BNx"])
    assert info["listed"] and lists is not None
    flat = [t for unit in lists for t in unit]
    assert sorted(flat) == list(range(n_gw + n_gx))
    for unit in lists:
        kinds = [t < n_gw for t in unit]            # True = GW
        assert kinds == sorted(kinds)               # all GX tiles first
    # no unit is left without work while another holds three tiles more
    sizes = [len(u) for u in lists[:min(units, n_gw + n_gx)]]
    assert min(sizes) >= 1


def test_tile_plan_without_a_table_for_very_many_tiles():
    info, lists = lbp.lbp_test_tile_plan(3072, 768, 400, 16, 8, 74, 1, 1)
    assert not info["listed"] and lists is None


def test_binding_structs_have_the_size_the_library_was_compiled_with():
    # a field added to include/lbp.h and not to the ctypes declarations (or the
    # other way round) would shift every field behind it
    from paper_2309_15275_b200 import binding as B
    lib = B._lib()
    for which, cls in ((0, B.Layer), (1, B.Extras), (2, B.View), (3, B.Basis)):
        assert lib.lbp_test_struct_size(which) == ctypes.sizeof(cls), cls.__name__
    assert lib.lbp_test_struct_size(99) == 0


@pytest.mark.parametrize("dtype", [0, 1])
def test_workspace_holds_the_coefficients_of_a_call_on_x_hat_at_full_rank(dtype):
    # at r = k^2 a call on x is Eq. 2, one on x_hat still writes g_y_hat and g_x_hat
    es = 2 if dtype == lbp.LBP_BF16 else 4
    for H, k in ((8, 4), (9, 4), (16, 8)):
        rows = 3 * (-(-H // k)) ** 2 * k * k
        got = lbp.lbp_workspace_bytes(3, H, H, 64, 96, k, dtype, lbp.LBP_F32, k * k)
        assert got >= rows * 96 * es + rows * 64 * 4


def test_module_forward_keeps_torch_dtype_rules():
    # y is matmul(x, W^T) + b under torch's own rules, also where the three types differ
    import torch
    lin = lbp.LbpLinear(16, 24, 4, [(0, 0)], bias=True)
    x = torch.randn(2, 4, 4, 16)

    def plain(x):
        return torch.matmul(x, lin.weight.t()) + lin.bias
    with torch.autocast("cpu", dtype=torch.bfloat16):
        y, want = lin(x), plain(x)
    assert y.dtype == want.dtype == torch.float32 and torch.equal(y, want)
    with torch.no_grad():
        lin.weight.data = lin.weight.data.bfloat16()   # bf16 weights and inputs, fp32 bias
        y, want = lin(x.bfloat16()), plain(x.bfloat16())
    assert y.dtype == want.dtype == torch.float32 and torch.equal(y, want)


@pytest.mark.parametrize("kind", ["numpy rows", "numpy scalars", "lists", "tensors", "floats", "none"])
def test_module_takes_bases_in_any_form_int_takes(kind):
    import numpy as np
    import torch
    pairs = [(0, 0), (0, 1), (1, 0)]
    bases = {"numpy rows": np.array(pairs), "numpy scalars": [(np.int64(i), np.int32(j)) for i, j in pairs],
             "lists": [list(p) for p in pairs], "tensors": [(torch.tensor(i), torch.tensor(j)) for i, j in pairs],
             "floats": [(float(i), float(j)) for i, j in pairs], "none": []}[kind]
    lin = lbp.LbpLinear(16, 24, 4, bases)
    x = torch.randn(2, 4, 4, 16)
    assert torch.equal(lin(x), torch.matmul(x, lin.weight.t()))


def test_batch_section_admits_one_thread_per_device():
    # the library's one stream and event set per device: what one batch call enqueues on
    # them is not interleaved with another thread's
    import threading
    import time
    lib = lbp.binding._lib()
    inside, most, order = [0, 0], [0, 0], threading.Lock()

    def enter(dev):
        def body(_):
            with order:
                inside[dev] += 1
                most[dev] = max(most[dev], inside[dev])
            time.sleep(0.02)
            with order:
                inside[dev] -= 1
            return 40 + dev
        cb = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p)(body)
        assert lib.lbp_test_side_section(dev, ctypes.cast(cb, ctypes.c_void_p), None) == 40 + dev
    threads = [threading.Thread(target=enter, args=(i % 2,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert most == [1, 1]


def test_kernel_attributes_are_set_on_every_device():
    import glob
    import os
    # the one place that sets them remembers the devices one by one
    devices = [0, 0, 1, 1, 0, 63, 63, 70, 70]
    done = (ctypes.c_uint8 * len(devices))()
    assert lbp.binding._lib().lbp_test_per_device((ctypes.c_int * len(devices))(*devices), len(devices), done) == 0
    assert list(done) == [1, 0, 1, 0, 0, 1, 0, 1, 1]
    csrc = os.path.join(os.path.dirname(lbp.__file__), "csrc")
    sites = [f for f in glob.glob(os.path.join(csrc, "*")) for _ in range(open(f).read().count("cudaFuncSetAttribute("))]
    assert [os.path.basename(f) for f in sites] == ["lbp_internal.h"]


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("ci,co,k,B,H", [(768, 3072, 8, 128, 16), (1024, 4096, 4, 128, 32), (64, 96, 4, 3, 9)])
def test_exact_backpropagation_on_x_needs_no_room_for_coefficients(dtype, ci, co, k, B, H):
    es = 2 if dtype == lbp.LBP_BF16 else 4
    rows = B * (-(-H // k) * k) ** 2
    size = lambda r, form: lbp.lbp_workspace_bytes(B, H, H, ci, co, k, dtype, lbp.LBP_F32, r, x_hat=form)  # noqa: E731
    ex = lambda form, **kw: lbp.lbp_workspace_bytes_ex(B, H, H, ci, co, k, dtype, lbp.LBP_F32, k * k, x_hat=form, **kw)  # noqa: E731
    # the status block and the fp32 planes of the K slices: 48 MiB for both at the most, beside g_W itself
    assert 256 <= size(k * k, False) <= 1024 + max(48 << 20, 192 * ci * co * 4 // max(1, (ci // 64) * (co // 128)))
    assert size(k * k, True) >= rows * (co * es + ci * 4)
    assert size(k * k, None) == max(size(k * k, False), size(k * k, True))
    assert size(2, False) == size(2, True) == size(2, None)
    # with extras: the same room on top of either
    assert ex(False, beta=1.0) - size(k * k, False) < 2 * ci * co * 4 + 8192
    assert ex(True, beta=1.0) - ex(False, beta=1.0) >= size(k * k, True) - size(k * k, False) - 4096


@pytest.mark.parametrize("Cin,Cout,B,H,W,k,r,n_extra,units,pair", [
    (768, 3072, 128, 16, 16, 8, 8, 0, 74, 1), (3072, 768, 128, 16, 16, 8, 16, 0, 37, 1),
    (768, 3072, 32, 14, 14, 16, 21, 32, 74, 1), (1280, 320, 36, 16, 16, 16, 1, 0, 74, 1),     # few large blocks
    (48, 192, 64, 56, 56, 8, 8, 0, 148, 0), (200, 72, 9, 7, 9, 4, 15, 300, 148, 0),
    (64, 64, 1, 8, 8, 8, 1, 1, 148, 0), (8, 8, 128, 8, 8, 8, 48, 0, 148, 0), (136, 520, 3, 17, 23, 8, 33, 5, 1, 1),
    (768, 3072, 32, 16, 16, 8, None, 0, 74, 1), (64, 64, 1, 1, 1, 4, None, 0, 148, 0), (136, 264, 1, 5, 13, 8, None, 0, 74, 1)])
def test_products_plan_covers_every_tile_once(Cin, Cout, B, H, W, k, r, n_extra, units, pair):
    # on the geometry of the kernel: channels of W along the tiles of g_x, whole blocks across
    bases = None if r is None else lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    info, lists = lbp.lbp_test_products_plan(B, H, W, Cin, Cout, k, bases, n_extra=n_extra, units=units, pair=pair)
    row_tile, most = (256, 256) if pair else (128, 128)
    blocks = 0 if r is None else B * -(-H // k) * -(-W // k)
    extra = B * H * W if r is None else n_extra
    assert info["BNw"] % (128 if pair else 64) == 0 and info["BNx"] % 32 == 0
    assert 0 < info["BNw"] <= most and 0 < info["BNx"] <= most
    assert 1 <= info["bpt"] and info["bpt"] * (r or 1) <= info["BNx"]
    assert info["num_kb_w"] == -(-blocks * (r or 1) // 64) + -(-extra // 64)
    assert info["kbps"] * info["splits"] >= info["num_kb_w"] > info["kbps"] * (info["splits"] - 1)
    assert info["splits"] == 1 or info["splits"] <= info["room"]
    n_gw = -(-Cout // row_tile) * -(-Cin // info["BNw"]) * info["splits"]
    n_gx = -(-Cin // row_tile) * (-(-blocks // info["bpt"]) + -(-extra // info["BNx"]))
    assert info["listed"] == (n_gw + n_gx <= 1536)
    if not info["listed"]:
        return
    assert sorted(t for unit in lists for t in unit) == list(range(n_gw + n_gx))
    for unit in lists:
        kinds = [t < n_gw for t in unit]            # True = GW
        assert kinds == sorted(kinds)               # all GX tiles first
    assert min(len(unit) for unit in lists[:n_gw + n_gx]) >= 1


@pytest.mark.parametrize("Cin,Cout,B,H,k,r", [
    (1024, 1024, 128, 64, 8, None), (256, 256, 512, 64, 8, None), (64, 64, 128, 64, 4, None), (4096, 1024, 128, 64, 8, 10),
    (3072, 768, 128, 16, 8, 16), (768, 3072, 128, 16, 8, 8)])
def test_planning_a_new_shape_is_quick(Cin, Cout, B, H, k, r):
    # searched inside the first call: a step per tile of a unit, not per tile and unit
    # (0.1 to 1 ms of a core; a second and more when every tile was weighed against every unit)
    import time
    bases = None if r is None else lbp.lbp_select_bases(k, lbp.SEL_PREFIX, r)
    spent = []
    for units in (74, 72, 70):      # a shape of its own each time
        t0 = time.process_time()
        lbp.lbp_test_products_plan(B, H, H, Cin, Cout, k, bases, units=units)
        spent.append(time.process_time() - t0)
    assert min(spent) < (0.015 if r is not None else 0.1), spent


def test_extras_keep_their_layout():
    # compiled callers: the size and the offsets of every field since the struct was first released
    from paper_2309_15275_b200 import binding as B
    at = {"beta": 0, "g_bias": 8, "n_extra": 16, "x_extra": 24, "gy_extra": 32, "gx_extra": 40, "x_view": 48,
          "gy_view": 72, "gx_view": 96, "x_extra_pitch": 120, "gy_extra_pitch": 128, "gx_extra_pitch": 136}
    assert {n: getattr(B.Extras, n).offset for n in at} == at
    assert B._lib().lbp_test_struct_size(1) == 144
    # what lies in the padding of such a caller's struct counts only with a bias
    lay = B._layer(1, 8, 8, 64, 64, 8, lbp.LBP_BF16, lbp.LBP_F32)
    ex = B.Extras(beta=1.0, g_bias_dtype=12345)
    assert B._lib().lbp_workspace_bytes_ex(ctypes.byref(lay), 8, ctypes.byref(ex)) > 0
    ex.g_bias = 16
    assert B._lib().lbp_workspace_bytes_ex(ctypes.byref(lay), 8, ctypes.byref(ex)) == 0


def test_another_torch_makes_the_binding_stale(monkeypatch):
    from paper_2309_15275_b200 import build
    build.build_library()
    assert not build._stale()
    monkeypatch.setattr(build, "_torch_version", lambda: "0.0.0+other")
    assert build._stale()


def test_module_attributes_and_operands_as_torch_takes_them():
    import torch

    class Tagged(torch.Tensor):
        pass
    lin = lbp.LbpLinear(16, 24, 4, [(0, 0)], bias=True)
    x = torch.randn(2, 4, 4, 16)
    want = lin(x)
    for bases in ([[0, 0], [0, 1]], np.array([[0, 0], [0, 1]]), ((0, 0),)):    # set after construction
        lin.bases = bases
        assert torch.equal(lin(x), want)
    lin.k = np.int64(4)
    assert torch.equal(lin(x), want)
    y = lin(x.as_subclass(Tagged))
    assert type(y) is Tagged and torch.equal(y.as_subclass(torch.Tensor), want)
    lin.grid = (np.int64(4), 4)
    assert torch.equal(lin(x.flatten(1, 2)), want.flatten(1, 2))
    for wrong in ([(0,)], [0, 1], 7, None, [("a", "b")]):
        lin.bases = wrong
        with pytest.raises(ValueError):
            lin(x.flatten(1, 2))


@pytest.mark.parametrize("ci,co,rows", [(64, 64, 5), (448, 1792, 640), (768, 3072, 32768), (8, 8, 2 ** 31 - 256),
                                        (8, 8, 2 ** 38)])
def test_fp32_products_are_planned_whatever_the_switch_says(monkeypatch, ci, co, rows):
    def plan(form, room):
        if form is None:
            monkeypatch.delenv("LBP_FP32_FORM", raising=False)
        else:
            monkeypatch.setenv("LBP_FP32_FORM", form)
        lbp.lbp_test_reload_env()
        return lbp.lbp_test_float_plan(ci, co, rows, room)
    try:
        for room in (0, 1 << 20, 2 ** 63):
            free = plan(None, room)
            assert all(plan(form, room) == free for form in ("3", "-1", "", "x", "1x", "10"))
            for form in range(3):
                got = plan(str(form), room)
                # sizes beyond a tensor map's coordinates are left to the form without one
                assert got["form"] == (form if rows < 2 ** 31 - 256 else 0)
                bk = 64 if got["form"] else 32
                for kb, items, K in ((got["gx_kb"], got["gx_items"], co), (got["gw_kb"], got["gw_items"], rows)):
                    assert kb >= 1 and items >= 1 and kb * items >= -(-K // bk) > kb * (items - 1)
                    assert items == 1 or room > 0
    finally:
        monkeypatch.undo()
        lbp.lbp_test_reload_env()
