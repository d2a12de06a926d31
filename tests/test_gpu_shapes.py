"""Shapes at the edges of the kernels' dispatch rules (partly filled tiles, remainders, smallest and largest of a range),
each against the float64 oracle."""
import pytest

from fbl_inputs import LayerConfig, MlpConfig, XattnConfig

import test_gpu_layer
import test_gpu_lora
import test_gpu_mlp
import test_gpu_xattn

pytestmark = pytest.mark.gpu


def check(cfg):
    if isinstance(cfg, MlpConfig):
        test_gpu_mlp.run_and_compare(cfg, guard_bytes=4096)
    elif isinstance(cfg, XattnConfig):
        test_gpu_xattn.run_and_compare(cfg, guard_bytes=4096)
    else:
        test_gpu_layer.run_and_compare(cfg, affine_noise=True, guard_bytes=4096)


@pytest.mark.parametrize("cfg", [
    # fewer token rows than one tile, one 64-wide key head, one memory tile beside many query rows
    LayerConfig("sh1", 1, 121, 128, 2, 1, 64, "bf16", "layernorm", True, True, True, 1e-5, 201, 0.05),
    LayerConfig("sh2", 3, 17, 192, 3, 1, 128, "bf16", "rmsnorm", False, False, False, 1e-5, 202, 0.05),
    LayerConfig("sh3", 2, 150, 320, 5, 1, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 203, 0.05),
    MlpConfig("sh4", 1, 40, 64, 192, "bf16", "layernorm", "swiglu", True, True, 1e-5, 204, 0.05),
    XattnConfig("sh5", 1, 130, 9, 128, 64, 2, 1, 64, "bf16", "layernorm", True, True, 1e-5, 205, 0.05),
], ids=lambda c: c.name)
def test_tensor_core_kernels_on_partly_filled_tiles(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # row widths of the norm kernels: part of a warp, a ragged last warp, several warps, more than one vector per thread
    # (fp32 above 2048 columns, bf16 above 4096); one, two and four rows per pass, with a short last block
    LayerConfig("nw1", 1, 9, 64, 1, 1, 64, "bf16", "layernorm", False, True, True, 1e-5, 211, 0.05),
    LayerConfig("nw2", 2, 613, 192, 2, 1, 64, "bf16", "rmsnorm", True, True, False, 1e-5, 212, 0.05),
    LayerConfig("nw3", 3, 401, 320, 2, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 213, 0.05),
    LayerConfig("nw4", 1, 70, 4160, 1, 1, 64, "bf16", "layernorm", False, False, True, 1e-5, 214, 0.02),
    LayerConfig("nw5", 2, 45, 96, 1, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 215, 0.1),
    LayerConfig("nw6", 1, 700, 160, 1, 1, 32, "fp32", "rmsnorm", False, True, False, 1e-5, 216, 0.1),
    LayerConfig("nw7", 1, 20, 2080, 1, 1, 32, "fp32", "layernorm", False, False, False, 1e-5, 217, 0.02),
], ids=lambda c: c.name)
def test_norm_row_widths(cfg):
    check(cfg)


@pytest.mark.parametrize("offset", [0, 1], ids=["aligned", "element-aligned"])
@pytest.mark.parametrize("b,t,d,dtype", [(1, 1, 64, "bf16"), (3, 13, 192, "bf16"), (2, 37, 96, "fp32"), (1, 9, 16384, "bf16"), (5, 130, 64, "fp32")])
def test_pack_and_unpack(b, t, d, dtype, offset):
    import torch
    from paper_2607_21624_b200 import LayerRunner
    from paper_2607_21624_b200.binding import TENSOR
    w = 64 if dtype == "bf16" else 32
    run = LayerRunner(LayerConfig("pk", b, t, d, 1, 1, w, dtype, "layernorm", True, False, False, 1e-5, 0, 0.02), guard_bytes=4096)
    n, stream, t_pad = b * t * d, torch.cuda.current_stream().cuda_stream, (t + 7) // 8 * 8
    src = torch.randn(n + 1, device="cuda").to(run.tdtype)[offset:offset + n]
    run.buf["X"].fill_(255)
    run.plan.pack(TENSOR["X"], src.data_ptr(), run.buf["X"].data_ptr(), stream)
    tiled = run.buf["X"].view(run.tdtype).view(d // w, b, t_pad, w)
    want = src.view(b, t, d // w, w).permute(2, 0, 1, 3)
    assert torch.equal(tiled[:, :, :t], want) and not tiled[:, :, t:].any()
    back = torch.full((n + 2,), 7.0, device="cuda").to(run.tdtype)
    run.plan.unpack(TENSOR["X"], run.buf["X"].data_ptr(), back[offset:].data_ptr(), stream)
    assert torch.equal(back[offset:offset + n], src) and (back[offset + n:] == 7).all() and (back[:offset] == 7).all()
    assert run.guards_intact() == []


@pytest.mark.parametrize("cfg", [
    # fp32 products: partly filled 64 x 64 tiles both ways, reductions of one to many 32-wide blocks (1 to 8 slices), all
    # operand orientations, heads of 32, 64 and 128
    LayerConfig("ff1", 1, 5, 32, 1, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 221, 0.2),
    LayerConfig("ff2", 3, 67, 160, 5, 1, 32, "fp32", "rmsnorm", True, True, False, 1e-5, 222, 0.1),
    LayerConfig("ff3", 2, 129, 1056, 3, 3, 64, "fp32", "layernorm", False, False, True, 1e-5, 223, 0.03),
    LayerConfig("ff4", 1, 200, 96, 2, 1, 128, "fp32", "rmsnorm", True, True, True, 1e-5, 224, 0.1),
    MlpConfig("ff5", 2, 70, 96, 416, "fp32", "layernorm", "swiglu", True, True, 1e-5, 225, 0.1),
    MlpConfig("ff6", 1, 1100, 64, 256, "fp32", "rmsnorm", "gelu", True, False, 1e-5, 226, 0.1),
    XattnConfig("ff7", 2, 33, 90, 64, 224, 4, 2, 32, "fp32", "layernorm", True, True, 1e-5, 227, 0.1),
], ids=lambda c: c.name)
def test_fp32_gemm_tiles_and_slices(cfg):
    check(cfg)


@pytest.mark.parametrize("slices", ["1", "2", "4", "8"])
@pytest.mark.parametrize("bn", ["64", "128"])
def test_fp32_products_on_every_tile(bn, slices, monkeypatch):
    # tiles that end in the middle of a panel both ways, reductions of fewer 64-column blocks than slices and of a half one at
    # the end, all operand orientations, fused row reduction, residual, padding rows
    monkeypatch.setenv("FBL_F32_BN", bn)
    monkeypatch.setenv("FBL_F32_SLICES", slices)
    check(LayerConfig("ft1", 3, 67, 160, 5, 1, 32, "fp32", "rmsnorm", True, True, True, 1e-5, 228, 0.1))
    check(LayerConfig("ft2", 1, 390, 352, 3, 3, 64, "fp32", "layernorm", False, False, False, 1e-5, 229, 0.05))


@pytest.mark.parametrize("cfg", [
    # fp32 attention on the tensor cores: its shortest sequences, tiles of 64 and 128 rows that end early, at their edge and one
    # past it on either side, grouped heads with one block and with a cluster to a key tile, both head widths, masks
    LayerConfig("fc1", 2, 33, 128, 2, 2, 64, "fp32", "layernorm", True, True, True, 1e-5, 232, 0.1),
    LayerConfig("fc2", 3, 65, 96, 4, 1, 32, "fp32", "rmsnorm", False, True, False, 1e-5, 233, 0.1),
    LayerConfig("fc3", 1, 128, 128, 2, 1, 64, "fp32", "layernorm", True, False, False, 1e-5, 234, 0.1),
    LayerConfig("fc4", 2, 129, 64, 3, 3, 32, "fp32", "rmsnorm", True, False, True, 1e-5, 235, 0.1),
    LayerConfig("fc5", 1, 450, 192, 6, 2, 64, "fp32", "layernorm", True, True, False, 1e-5, 236, 0.1),
    LayerConfig("fc6", 70, 192, 64, 3, 1, 64, "fp32", "layernorm", False, False, False, 1e-5, 237, 0.1),
    XattnConfig("fc7", 2, 9, 200, 96, 64, 4, 2, 32, "fp32", "layernorm", True, True, 1e-5, 238, 0.1),
    XattnConfig("fc8", 1, 260, 7, 64, 96, 2, 1, 64, "fp32", "rmsnorm", False, True, 1e-5, 239, 0.1),
], ids=lambda c: c.name)
def test_fp32_attention_on_tensor_cores(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    XattnConfig("fm1", 96, 80, 16, 128, 128, 8, 8, 64, "fp32", "layernorm", False, True, 1e-5, 246, 0.1),
    XattnConfig("fm2", 75, 70, 32, 128, 64, 4, 1, 64, "fp32", "rmsnorm", True, False, 1e-5, 247, 0.1),
    XattnConfig("fm3", 74, 70, 32, 128, 64, 4, 1, 64, "fp32", "rmsnorm", True, False, 1e-5, 248, 0.1),
], ids=lambda c: c.name)
def test_fp32_attention_of_few_memory_rows(cfg):
    # either side of the line between the two kernel families; neither takes longer than multiply-adds alone
    import torch
    from paper_2607_21624_b200 import XattnRunner
    check(cfg)
    us = {}
    for path in (0, 1):
        run = XattnRunner(cfg)
        run.plan.set_kernel_path(path)
        run.plan.profile_enable(True)
        times = []
        for _ in range(20):
            total = 0.0
            for part in (run.forward, run.backward):
                part()
                torch.cuda.synchronize()
                total += sum(ms for name, ms in run.plan.profile_read() if name.startswith("attn"))
            times.append(total)
        us[path] = sorted(times)[10] * 1e3
    assert us[0] <= 1.1 * us[1] + 2, us


@pytest.mark.parametrize("head_dim", [32, 64])
def test_fp32_attention_of_operands_without_parts(head_dim):
    # infinities among V and among dA: the same results as plain multiply-adds, and finite columns stay finite
    import numpy as np
    from fbl_inputs import make_inputs
    from paper_2607_21624_b200 import LayerRunner
    cfg = LayerConfig("fi1", 2, 150, 128, 4, 2, head_dim, "fp32", "layernorm", False, True, False, 1e-5, 240, 0.1)
    inp = dict(make_inputs(cfg, affine_noise=True))
    outs = {}
    for path in (0, 1):
        for case in ("V", "dA"):
            run = LayerRunner(cfg, guard_bytes=4096)
            run.plan.set_kernel_path(path)
            changed = dict(inp)
            if case == "V":
                changed["bv"] = np.array(inp["bv"], copy=True)
                changed["bv"][5], changed["bv"][head_dim + 9] = np.inf, -np.inf
            else:
                changed["dY"] = np.array(inp["dY"], copy=True)
                changed["dY"].reshape(-1, cfg.d_model)[200, 7] = np.inf     # dA of one token is infinite
            run.load_inputs(changed)
            run.step()
            assert run.status() == 0 and run.guards_intact() == []
            outs[path, case] = {n: np.asarray(run.saved_view(n), dtype=np.float64) for n in ("A", "LSE", "dA", "dQ", "dK", "dV")}
    for case, names in (("V", ("A", "LSE")), ("dA", ("A", "LSE", "dA", "dQ", "dK", "dV"))):
        for n in names:
            got, want = outs[0, case][n], outs[1, case][n]
            assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want)), (case, n)
            assert np.array_equal(got[np.isinf(got)], want[np.isinf(want)]), (case, n)
            m = np.isfinite(want)
            if not m.any():
                continue
            scale = np.abs(want[m]).max()
            assert np.linalg.norm((got[m] - want[m]) / scale) <= 1e-5 * np.linalg.norm(want[m] / scale), (case, n)
    assert np.isinf(outs[1, "V"]["A"]).any() and not np.isfinite(outs[1, "dA"]["dA"]).all()


@pytest.mark.parametrize("cfg", [
    LayerConfig("np1", 2, 150, 128, 4, 2, 64, "fp32", "layernorm", True, True, False, 1e-5, 241, 0.1),
    LayerConfig("np2", 1, 333, 96, 6, 6, 32, "fp32", "rmsnorm", True, False, True, 1e-5, 242, 0.1),
], ids=lambda c: c.name)
def test_fp32_attention_of_an_infinite_token_under_a_mask(cfg):
    # one token infinite in Q, K and V: the queries before it are what they are without it
    import numpy as np
    from fbl_inputs import make_inputs
    from paper_2607_21624_b200 import LayerRunner
    inp, at = dict(make_inputs(cfg, affine_noise=True)), 70
    outs = []
    for poison in (False, True):
        run = LayerRunner(cfg, guard_bytes=4096)
        X = np.array(inp["X"], copy=True)
        if poison:
            X[0, at, 3] = np.inf
        run.load_inputs(dict(inp, X=X))
        run.step()
        assert run.status() == 0 and run.guards_intact() == []
        outs.append({n: np.asarray(run.saved_view(n), dtype=np.float64) for n in ("A", "LSE", "dQ")})
    clean, got = outs
    for n in ("A", "dQ"):
        assert not np.isfinite(got[n][0, at:]).any(), n
        assert np.linalg.norm(got[n][0, :at] - clean[n][0, :at]) <= 1e-5 * np.linalg.norm(clean[n][0, :at]), n
        assert np.linalg.norm(got[n][1:] - clean[n][1:]) <= 1e-5 * np.linalg.norm(clean[n][1:]), n
    assert np.abs(got["LSE"][0, :, :at] - clean["LSE"][0, :, :at]).max() <= 1e-5 * np.abs(clean["LSE"]).max()


@pytest.mark.parametrize("cfg", [
    LayerConfig("nt1", 4, 197, 768, 12, 12, 64, "fp32", "layernorm", False, True, True, 1e-6, 243, 0.02),
    LayerConfig("nt2", 1, 1024, 512, 16, 4, 32, "fp32", "layernorm", True, False, True, 1e-6, 244, 0.02),
    MlpConfig("nt3", 2, 400, 512, 2048, "fp32", "layernorm", "gelu", True, True, 1e-6, 245, 0.02),
], ids=lambda c: c.name)
def test_fp32_steps_with_an_infinity_take_no_other_time(cfg):
    # an infinity reaches every weight gradient; the step must stay within a small factor of the multiply-adds that it falls
    # back to (with a thread to a result it took 25 to 53 times as long)
    import torch
    from paper_2607_21624_b200 import LayerRunner, MlpRunner
    us = {}
    for path in (0, 1):
        run = MlpRunner(cfg) if isinstance(cfg, MlpConfig) else LayerRunner(cfg)
        run.plan.set_kernel_path(path)
        for n, b in run.buf.items():
            b.view(run.tdtype).normal_(std=0.02 if n[0] == "W" else 1.0)
        run.vec["gamma"].fill_(1.0)
        run.buf["X"].view(run.tdtype)[1000] = float("inf")
        for _ in range(3):
            run.step()
        first, last = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        first.record()
        for _ in range(5):
            run.step()
        last.record()
        assert run.status() == 0
        us[path] = first.elapsed_time(last) * 200
        assert not torch.isfinite(run.buf["dW1" if isinstance(cfg, MlpConfig) else "dWq"].view(run.tdtype)).all()
    assert us[0] <= 4 * us[1], us


def _mlp_outputs(cfg, inp, path):
    import numpy as np
    from paper_2607_21624_b200.mlp import MlpRunner
    run = MlpRunner(cfg, guard_bytes=4096)
    run.plan.set_kernel_path(path)
    run.load_inputs(inp)
    run.step()
    assert run.status() == 0 and run.guards_intact() == []
    return {n: np.asarray(run.fetch(n), dtype=np.float64) for n in ("Y", "dX", "dW1", "dW2", "db1", "db2", "dgamma")}


def test_fp32_products_are_no_further_off_than_multiply_adds():
    # against 64 bits; both kernels' sums are within a few units of the last place, so no element-wise bound is tighter than this
    import numpy as np
    from fbl_inputs import make_mlp_inputs
    from oracle import mlp as orc
    cfg = MlpConfig("fa1", 2, 300, 512, 768, "fp32", "layernorm", "gelu", True, False, 1e-5, 230, 0.05)
    inp = make_mlp_inputs(cfg, affine_noise=True)
    Y, _, grads = orc.mlp_fwd_bwd(cfg, inp)
    ref = dict(grads, Y=Y)
    off = lambda got, n: np.linalg.norm(got[n] - ref[n]) / np.linalg.norm(ref[n])
    default, ffma = (_mlp_outputs(cfg, inp, path) for path in (0, 1))
    for n in ("Y", "dX", "dW1", "dW2"):
        assert off(default, n) <= off(ffma, n), (n, off(default, n), off(ffma, n))


def test_fp32_products_of_operands_without_parts():
    # infinities, NaN, and values that round to infinity in bf16: the same results as plain multiply-adds
    import numpy as np
    from fbl_inputs import make_mlp_inputs
    cfg = MlpConfig("fa2", 1, 150, 160, 192, "fp32", "rmsnorm", "gelu", True, False, 1e-5, 231, 0.05)
    inp = dict(make_mlp_inputs(cfg, affine_noise=True))
    for n in ("W2", "dY"):
        inp[n] = np.array(inp[n], copy=True)
    inp["W2"][3, 5], inp["W2"][9, 7], inp["W2"][70, 130] = np.inf, -np.inf, 3.395e38
    flat = inp["dY"].reshape(-1, cfg.d_model)
    flat[11, 40], flat[77, 2] = np.nan, np.inf
    default, ffma = (_mlp_outputs(cfg, inp, path) for path in (0, 1))
    for n, want in ffma.items():
        got = default[n]
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want)), n
        assert np.array_equal(got[np.isinf(got)], want[np.isinf(want)]), n
        m = np.isfinite(want)
        if m.any():
            assert np.linalg.norm((got[m] - want[m]) / np.abs(want[m]).max()) <= 1e-5 * np.linalg.norm(want[m] / np.abs(want[m]).max()), n
    assert np.isinf(ffma["Y"]).any() and np.isfinite(ffma["Y"]).any()


@pytest.mark.parametrize("pair", ["-1", "1"], ids=["by-cost", "pairs"])
@pytest.mark.parametrize("cfg", [
    # columns that are not whole tiles, on every tile shape: one to a few tiles of rows, an odd number of 64-wide panels
    LayerConfig("rg1", 1, 300, 192, 5, 1, 64, "bf16", "layernorm", True, True, True, 1e-5, 241, 0.05),
    LayerConfig("rg2", 2, 500, 1088, 17, 17, 64, "bf16", "rmsnorm", True, False, False, 1e-5, 242, 0.02),
    MlpConfig("rg3", 3, 333, 448, 1216, "bf16", "layernorm", "gelu", True, True, 1e-5, 243, 0.03),
    # activations with two outputs, and the rotary embedding (both head widths, with biases), in the projections' epilogues
    MlpConfig("rg4", 2, 300, 256, 704, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 244, 0.03),
    LayerConfig("rg5", 2, 300, 192, 5, 1, 64, "bf16", "rmsnorm", True, True, True, 1e-5, 245, 0.01, 0.0, 10000.0),
    LayerConfig("rg6", 2, 141, 256, 3, 1, 128, "bf16", "layernorm", False, True, False, 1e-5, 246, 0.01, 0.0, 500.0),
    LayerConfig("rg7", 3, 77, 256, 3, 3, 64, "bf16", "layernorm", True, True, False, 1e-5, 247, 0.01, 0.0, 500.0),
], ids=lambda c: getattr(c, "name", ""))
def test_ragged_columns_on_every_gemm_tile(cfg, pair, monkeypatch):
    monkeypatch.setenv("FBL_GEMM_PAIR", pair)
    check(cfg)


def test_bands_of_row_tiles(monkeypatch):
    # CTA pairs: 17 row tiles are two bands of eight and one of a single, partly filled tile; several column tiles
    monkeypatch.setenv("FBL_GEMM_PAIR", "1")
    check(MlpConfig("rb1", 1, 4300, 192, 576, "bf16", "rmsnorm", "gelu", False, True, 1e-5, 248, 0.05))


@pytest.mark.parametrize("cfg", [
    # one key tile (dQ straight from the block), with one and several query tiles, grouped heads, both head widths
    LayerConfig("sa1", 2, 128, 128, 4, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 251, 0.05),
    LayerConfig("sa2", 2, 97, 256, 2, 1, 128, "bf16", "rmsnorm", False, False, False, 1e-5, 252, 0.05),
    XattnConfig("sa3", 2, 300, 120, 128, 64, 2, 1, 64, "bf16", "layernorm", True, True, 1e-5, 253, 0.05),
    XattnConfig("sa4", 1, 129, 33, 128, 64, 2, 1, 128, "bf16", "layernorm", False, True, 1e-5, 254, 0.05),
    # two key tiles and one or two query tiles in one block: full, ragged at either end, causal and not; then one past it
    LayerConfig("sa5", 2, 256, 128, 2, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 255, 0.05),
    LayerConfig("sa6", 2, 129, 192, 3, 3, 64, "bf16", "rmsnorm", True, False, False, 1e-5, 256, 0.05),
    LayerConfig("sa7", 3, 255, 128, 2, 2, 64, "bf16", "layernorm", False, True, False, 1e-5, 257, 0.05),
    LayerConfig("sa8", 2, 131, 128, 2, 2, 64, "bf16", "layernorm", False, False, True, 1e-5, 258, 0.05),
    XattnConfig("sa9", 2, 60, 200, 128, 64, 2, 2, 64, "bf16", "layernorm", True, True, 1e-5, 259, 0.05),
    XattnConfig("sa10", 2, 256, 130, 128, 192, 2, 2, 64, "bf16", "rmsnorm", True, True, 1e-5, 260, 0.05),
    LayerConfig("sa11", 2, 257, 128, 2, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 261, 0.05),
    XattnConfig("sa12", 2, 257, 256, 128, 64, 2, 2, 64, "bf16", "layernorm", True, True, 1e-5, 262, 0.05),
], ids=lambda c: c.name)
def test_attention_backward_of_short_sequences(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # fp32 attention: one to many 32-row tiles, 64-key / 64-query tiles full, half and ragged, groups, all head widths
    LayerConfig("fa1", 2, 33, 64, 2, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 271, 0.2),
    LayerConfig("fa2", 1, 224, 64, 2, 2, 64, "fp32", "rmsnorm", True, False, False, 1e-5, 272, 0.1),
    LayerConfig("fa3", 2, 161, 64, 4, 2, 64, "fp32", "layernorm", False, True, True, 1e-5, 273, 0.1),
    LayerConfig("fa4", 2, 117, 64, 2, 1, 128, "fp32", "layernorm", True, True, False, 1e-5, 274, 0.1),
    XattnConfig("fa5", 2, 97, 31, 64, 96, 2, 2, 128, "fp32", "layernorm", True, True, 1e-5, 275, 0.1),
    XattnConfig("fa6", 2, 1, 130, 64, 64, 2, 1, 64, "fp32", "rmsnorm", True, True, 1e-5, 276, 0.1),
], ids=lambda c: c.name)
def test_fp32_attention_tiles(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # few tokens and long reductions (cluster-split products): one to four row groups of a tile, two row tiles, remainders of
    # the reduction over the slices, every epilogue (bias, residual, row reduction, activations, rotation at both widths)
    LayerConfig("sp1", 1, 20, 1024, 16, 4, 64, "bf16", "layernorm", True, True, True, 1e-5, 281, 0.02),
    LayerConfig("sp2", 3, 50, 1088, 7, 7, 128, "bf16", "rmsnorm", True, True, False, 1e-5, 282, 0.02, 0.0, 10000.0),
    LayerConfig("sp3", 1, 101, 1216, 19, 1, 64, "bf16", "rmsnorm", False, False, True, 1e-5, 283, 0.02, 0.0, 10000.0),
    MlpConfig("sp4", 1, 33, 1024, 2048, "bf16", "layernorm", "gelu", True, True, 1e-5, 284, 0.02),
    MlpConfig("sp5", 2, 60, 1152, 1984, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 285, 0.02),
    # short reductions (128 x 64 tiles): one panel, a ragged number of panels, tiles up to the number of SMs
    LayerConfig("sp7", 2, 70, 448, 7, 7, 64, "bf16", "layernorm", True, True, True, 1e-5, 287, 0.02, 0.0, 10000.0),
    MlpConfig("sp8", 3, 129, 192, 576, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 288, 0.02),
    LayerConfig("sp9", 4, 250, 320, 5, 1, 64, "bf16", "rmsnorm", False, True, True, 1e-5, 289, 0.02),
    XattnConfig("sp6", 2, 9, 60, 1024, 1280, 8, 8, 128, "bf16", "layernorm", True, True, 1e-5, 286, 0.02),
], ids=lambda c: c.name)
def test_few_tokens_long_reductions(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # bias gradients summed beside the last products: ragged last slabs, one to three matrices' worth of pieces per block
    LayerConfig("cs1", 2, 290, 2048, 16, 16, 128, "bf16", "layernorm", True, True, True, 1e-5, 291, 0.01),
    LayerConfig("cs2", 9, 133, 1024, 16, 4, 64, "bf16", "rmsnorm", False, True, False, 1e-5, 292, 0.01, 0.0, 10000.0),
    MlpConfig("cs3", 2, 270, 1024, 4096, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 293, 0.01),
    MlpConfig("cs4", 5, 405, 768, 2048, "bf16", "layernorm", "gelu", True, False, 1e-5, 294, 0.01),
    XattnConfig("cs5", 1, 8, 520, 512, 512, 8, 8, 64, "bf16", "layernorm", True, True, 1e-5, 295, 0.02),
    XattnConfig("cs6", 2, 300, 300, 512, 256, 4, 4, 128, "bf16", "rmsnorm", True, True, 1e-5, 296, 0.02),
], ids=lambda c: c.name)
def test_bias_gradients_beside_products(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # fp32 attention backward with a key tile's items dealt over 2, 4 and 8 blocks: fewer items than blocks (causal ends),
    # uneven shares, a ragged key tile, every head width
    LayerConfig("fs1", 1, 70, 128, 4, 1, 32, "fp32", "layernorm", True, False, False, 1e-5, 301, 0.05),
    LayerConfig("fs2", 2, 129, 128, 6, 2, 64, "fp32", "rmsnorm", False, False, True, 1e-5, 302, 0.05),
    LayerConfig("fs3", 1, 100, 256, 3, 1, 128, "fp32", "rmsnorm", True, True, True, 1e-5, 303, 0.05, 0.0, 10000.0),
    XattnConfig("fs4", 1, 150, 41, 96, 128, 3, 1, 64, "fp32", "layernorm", True, True, 1e-5, 304, 0.05),
    XattnConfig("fs5", 3, 40, 33, 128, 64, 2, 1, 32, "fp32", "rmsnorm", False, False, 1e-5, 305, 0.05),
], ids=lambda c: c.name)
def test_fp32_attention_backward_slices(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # the multiply-add kernels, which the tensor-core ones are compared with: products on partly filled 64 x 64 tiles, one to eight
    # slices of a reduction, all operand orientations; attention of one to many tiles, groups, items dealt over a cluster
    LayerConfig("ma1", 1, 5, 32, 1, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 431, 0.2),
    LayerConfig("ma2", 3, 67, 160, 5, 1, 32, "fp32", "rmsnorm", True, True, False, 1e-5, 432, 0.1),
    LayerConfig("ma3", 2, 129, 1056, 3, 3, 64, "fp32", "layernorm", False, False, True, 1e-5, 433, 0.03),
    LayerConfig("ma4", 1, 224, 64, 2, 2, 64, "fp32", "rmsnorm", True, False, False, 1e-5, 434, 0.1),
    LayerConfig("ma5", 2, 129, 128, 6, 2, 64, "fp32", "rmsnorm", False, False, True, 1e-5, 435, 0.05),
    LayerConfig("ma6", 1, 70, 128, 4, 1, 32, "fp32", "layernorm", True, False, False, 1e-5, 436, 0.05, 0.0, 10000.0),
    MlpConfig("ma7", 2, 70, 96, 416, "fp32", "layernorm", "swiglu", True, True, 1e-5, 437, 0.1),
    MlpConfig("ma8", 1, 1100, 64, 256, "fp32", "rmsnorm", "gelu", True, False, 1e-5, 438, 0.1),
    XattnConfig("ma9", 2, 33, 90, 64, 224, 4, 2, 32, "fp32", "layernorm", True, True, 1e-5, 439, 0.1),
    XattnConfig("ma10", 1, 150, 41, 96, 128, 3, 1, 64, "fp32", "layernorm", True, True, 1e-5, 440, 0.05),
], ids=lambda c: c.name)
def test_fp32_multiply_add_kernels(cfg):
    compare = test_gpu_mlp if isinstance(cfg, MlpConfig) else test_gpu_xattn if isinstance(cfg, XattnConfig) else test_gpu_layer
    compare.run_and_compare(cfg, affine_noise=True, path=1, guard_bytes=4096)


@pytest.mark.parametrize("cfg", [
    # tensor-core attention backward with a key tile's items dealt over 2, 4 and 8 blocks: shares that do not divide, blocks
    # without items (causal ends), one key tile (dQ written at once), ragged key tiles, the rotation behind it
    LayerConfig("bs1", 1, 300, 256, 8, 1, 64, "bf16", "layernorm", True, False, False, 1e-5, 311, 0.02),
    LayerConfig("bs2", 1, 420, 256, 5, 1, 128, "bf16", "rmsnorm", True, False, True, 1e-5, 312, 0.02, 0.0, 10000.0),
    LayerConfig("bs3", 2, 100, 256, 12, 2, 64, "bf16", "layernorm", False, True, True, 1e-5, 313, 0.02),
    LayerConfig("bs4", 1, 77, 256, 9, 1, 128, "bf16", "rmsnorm", True, False, True, 1e-5, 314, 0.02),
    XattnConfig("bs5", 1, 640, 140, 256, 128, 3, 1, 64, "bf16", "layernorm", True, True, 1e-5, 315, 0.02),
    XattnConfig("bs6", 3, 257, 520, 256, 128, 2, 1, 128, "bf16", "rmsnorm", False, False, 1e-5, 316, 0.02),
], ids=lambda c: c.name)
def test_attention_backward_slices(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # cluster-split products with reductions of nine k-blocks, which four blocks do not share evenly, beside longer ones: the
    # weight gradients of one launch or the other, the norm's output gradient, an adapter step's, both feed-forward forms
    LayerConfig("ns1", 1, 520, 1536, 2, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 321, 0.02),
    LayerConfig("ns2", 1, 576, 256, 8, 8, 64, "bf16", "layernorm", True, True, True, 1e-5, 322, 0.02),
    LayerConfig("ns3", 7, 197, 192, 3, 3, 64, "bf16", "layernorm", False, True, True, 1e-5, 323, 0.02),
    (LayerConfig("ns4", 1, 1345, 128, 2, 2, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 324, 0.02), 16),
    MlpConfig("ns5", 1, 520, 256, 1536, "bf16", "layernorm", "gelu", True, True, 1e-5, 325, 0.02),
    MlpConfig("ns6", 1, 576, 128, 1024, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 326, 0.02),
    XattnConfig("ns7", 1, 520, 64, 1536, 64, 2, 2, 64, "bf16", "layernorm", True, True, 1e-5, 327, 0.02),
], ids=lambda c: getattr(c, "name", "ns4"))
def test_cluster_slices_of_nine_k_blocks(cfg):
    if isinstance(cfg, tuple):
        test_gpu_lora.run_and_compare(cfg[0], cfg[1], guard_bytes=4096)
    else:
        check(cfg)


@pytest.mark.parametrize("cfg", [
    # less than a tile of token rows on either side, both head widths, groups, one and several key tiles
    LayerConfig("fp1", 1, 50, 128, 4, 4, 64, "bf16", "layernorm", False, True, True, 1e-5, 331, 0.1),
    LayerConfig("fp2", 3, 40, 256, 4, 2, 128, "bf16", "rmsnorm", False, False, False, 1e-5, 332, 0.1),
    XattnConfig("fp3", 2, 9, 300, 128, 192, 4, 2, 64, "bf16", "layernorm", True, True, 1e-5, 333, 0.1),
    XattnConfig("fp4", 1, 300, 70, 128, 64, 3, 1, 128, "bf16", "rmsnorm", False, True, 1e-5, 334, 0.1),
], ids=lambda c: c.name)
def test_few_rows_keep_fp32_probabilities(cfg):
    # A, dQ, dK, dV from the stored operands in 64 bits, rounded once, are what the kernels store: fp32 sums of a few hundred
    # terms are within about 1e-5 of the terms' size, 1 % of the spacing of bf16 values, so they round elsewhere in about 1 %
    # of the elements; P and dS in bf16 (2e-3 per term) move a fifth of them
    import numpy as np
    import torch
    run = (test_gpu_xattn if isinstance(cfg, XattnConfig) else test_gpu_layer).run_and_compare(cfg, guard_bytes=4096)
    hd, hq, hkv = cfg.head_dim, cfg.n_q_heads, cfg.n_kv_heads
    heads = lambda n, h: run.saved_view(n).reshape(cfg.batch, -1, h, hd).transpose(0, 2, 1, 3)
    Q, dA = heads("Q", hq), heads("dA", hq)
    K, V = (np.repeat(heads(n, hkv), hq // hkv, 1) for n in "KV")
    S = Q @ K.swapaxes(2, 3) / np.sqrt(hd)
    P = np.exp(S - S.max(-1, keepdims=True))
    P /= P.sum(-1, keepdims=True)
    dS = P * (dA @ V.swapaxes(2, 3) - run.saved_view("D")[..., None]) / np.sqrt(hd)
    group = lambda x: x.reshape(cfg.batch, hkv, hq // hkv, *x.shape[2:]).sum(2)
    for name, want in (("A", P @ V), ("dQ", dS @ K), ("dK", group(dS.swapaxes(2, 3) @ Q)), ("dV", group(P.swapaxes(2, 3) @ dA))):
        rounded = torch.from_numpy(want).to(torch.bfloat16).double().numpy()
        same = (rounded == heads(name, want.shape[1])).mean()
        print(name, same)
        assert same >= 0.97, (name, same)


@pytest.mark.parametrize("cfg", [
    # one or two query tiles a block of the forward: pairs of five causal tiles, tiles that just do not and just do fit the SMs at
    # once, few key tiles, a round of pairs too many, long causal chains
    LayerConfig("qt1", 13, 520, 256, 4, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 361, 0.05),
    LayerConfig("qt2", 15, 515, 128, 2, 1, 64, "bf16", "rmsnorm", False, False, False, 1e-5, 362, 0.05),
    LayerConfig("qt3", 1, 300, 256, 4, 4, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 363, 0.05),
    LayerConfig("qt4", 13, 520, 256, 4, 4, 64, "bf16", "rmsnorm", False, False, True, 1e-5, 364, 0.05),
    LayerConfig("qt5", 11, 900, 128, 2, 1, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 365, 0.05),
    XattnConfig("qt6", 10, 700, 200, 256, 128, 4, 2, 64, "bf16", "layernorm", True, True, 1e-5, 366, 0.05),
], ids=lambda c: c.name)
def test_query_tiles_of_a_forward_block(cfg):
    check(cfg)


@pytest.mark.parametrize("cfg", [
    # a key and a query tile that reach past a sequence: fp32 at each head width and beside a cluster, bf16 of few rows
    LayerConfig("iso1", 3, 20, 64, 2, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 341, 0.2),
    LayerConfig("iso2", 3, 77, 128, 4, 2, 64, "fp32", "rmsnorm", False, False, True, 1e-5, 342, 0.1),
    LayerConfig("iso3", 3, 41, 128, 8, 1, 128, "fp32", "rmsnorm", True, False, False, 1e-5, 343, 0.1),
    LayerConfig("iso4", 3, 30, 128, 4, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 344, 0.1),
    LayerConfig("iso5", 3, 33, 128, 2, 2, 128, "bf16", "rmsnorm", False, False, True, 1e-5, 345, 0.1),
    XattnConfig("iso6", 3, 9, 50, 128, 64, 2, 1, 64, "bf16", "layernorm", True, True, 1e-5, 346, 0.1),
    XattnConfig("iso7", 3, 50, 70, 64, 96, 2, 2, 64, "fp32", "layernorm", True, True, 1e-5, 347, 0.1),
], ids=lambda c: c.name)
def test_values_that_are_not_finite_stay_in_their_sequence(cfg):
    import numpy as np
    from fbl_inputs import make_inputs, make_xattn_inputs
    from paper_2607_21624_b200 import LayerRunner, XattnRunner
    cross = isinstance(cfg, XattnConfig)
    inp = (make_xattn_inputs if cross else make_inputs)(cfg)
    run = (XattnRunner if cross else LayerRunner)(cfg)
    names = ("Y", "dX", "dM") if cross else ("Y", "dX")
    run.load_inputs(inp)
    run.step()
    plain = {n: run.fetch(n) for n in names}
    for n in ("X", "M") if cross else ("X",):
        inp[n][1] = np.inf
    run.load_inputs(inp)
    run.step()
    assert run.status() == 0
    for n in names:
        got = run.fetch(n)
        assert not np.isfinite(got[1]).any(), n
        for b in (0, 2):                  # the same sums, in an order that dQ's additions may change in the last place
            assert np.abs(got[b] - plain[n][b]).max() <= (1e-5 if cfg.dtype == "fp32" else 1e-2) * np.abs(plain[n][b]).max(), (n, b)


@pytest.mark.parametrize("rows,cols", [(8, 64), (2048, 768), (1000, 4096)])
def test_early_sums_wait_behind_a_launch_that_vouches_for_nothing(rows, cols):
    import ctypes as C
    import torch
    from paper_2607_21624_b200.binding import Plan, _check, aligned_bytes, desc_from_config, lib
    plan = Plan(desc_from_config(LayerConfig("eo", 1, 64, 64, 1, 1, 64, "bf16", "layernorm", True, True, False, 1e-5, 0, 0.02)))
    fn = lib().fbl_selftest_early_order
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_int64, C.c_int64, C.c_void_p, C.c_void_p, C.c_void_p]
    dev = torch.device("cuda:0")
    m = aligned_bytes(torch, rows * cols * 2, dev)
    scratch = aligned_bytes(torch, 1024 + plan.colsum_scratch_bytes(rows, cols), dev)
    out = torch.zeros(cols, device=dev)
    for _ in range(3):
        m.zero_()
        out.zero_()
        _check(fn(plan._h, m.data_ptr(), rows, cols, out.data_ptr(), scratch.data_ptr(), torch.cuda.current_stream().cuda_stream))
        assert (out == rows).all()


@pytest.mark.parametrize("cfg", [
    LayerConfig("bs1", 2, 60, 256, 4, 2, 64, "bf16", "layernorm", True, True, True, 1e-5, 351, 0.05),
    LayerConfig("bs2", 2, 300, 256, 4, 2, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 352, 0.05, 0.0, 10000.0),
    LayerConfig("bs3", 1, 70, 64, 2, 1, 32, "fp32", "layernorm", True, True, True, 1e-5, 353, 0.1),
    MlpConfig("bs4", 1, 200, 256, 704, "bf16", "rmsnorm", "swiglu", True, True, 1e-5, 354, 0.05),
    XattnConfig("bs5", 1, 140, 200, 128, 192, 2, 2, 64, "bf16", "layernorm", True, True, 1e-5, 355, 0.05),
], ids=lambda c: c.name)
def test_one_plan_over_many_sets_of_buffers(cfg):
    # a model's layers share a plan: each pass goes to the buffers it is called with, whichever were before
    import dataclasses
    import numpy as np
    from fbl_inputs import make_inputs, make_mlp_inputs, make_xattn_inputs
    from paper_2607_21624_b200 import LayerRunner, MlpRunner, XattnRunner
    make, Runner = (make_mlp_inputs, MlpRunner) if isinstance(cfg, MlpConfig) else (make_xattn_inputs, XattnRunner) if \
        isinstance(cfg, XattnConfig) else (make_inputs, LayerRunner)
    inputs = [make(dataclasses.replace(cfg, seed=cfg.seed + 1000 * i)) for i in range(4)]
    alone = [Runner(cfg) for _ in inputs]
    shared = [Runner(cfg) for _ in inputs]
    for a, s, inp in zip(alone, shared, inputs):
        a.load_inputs(inp)
        s.load_inputs(inp)
        a.step()
    for s in shared:
        s.plan = shared[0].plan
    for order in ((0, 1, 2, 3), (3, 1, 0, 2)):
        for i in order:
            shared[i].step()
    for a, s in zip(alone, shared):
        assert s.status() == 0
        for n in a.OUT_MATS:
            if n in a.buf:                  # dQ's additions may come in another order
                want = a.fetch(n)
                assert np.abs(s.fetch(n) - want).max() <= (1e-5 if cfg.dtype == "fp32" else 1e-2) * np.abs(want).max(), n
