"""fp32 on the tensor cores, whose operands are three bf16 parts each, against what fp32 arithmetic gives: the ends of the range and
results that are exact."""
import numpy as np
import pytest

from fbl_inputs import LayerConfig, XattnConfig, make_inputs, make_xattn_inputs
from paper_2607_21624_b200 import LayerRunner, XattnRunner

pytestmark = pytest.mark.gpu


def outputs(cfg, inp, path, names):
    run = (XattnRunner if isinstance(cfg, XattnConfig) else LayerRunner)(cfg, guard_bytes=4096)
    run.plan.set_kernel_path(path)
    run.load_inputs(inp)
    run.step()
    assert run.status() == 0 and run.guards_intact() == []
    return {n: run.fetch(n) if n in run.OUT_MATS else np.asarray(run.saved_view(n), dtype=np.float64) for n in names}


def off(got, want):
    return np.linalg.norm(got - want) / np.linalg.norm(want)


@pytest.mark.parametrize("head_dim", [32, 64])
def test_scores_below_the_range(head_dim):
    # one key so large that its scores are minus infinity, its parts' products infinities of both signs: its weight is zero
    cfg = XattnConfig("fr1", 1, 70, 100, 128, 64, 2, 64 // head_dim, head_dim, "fp32", "rmsnorm", True, False, 1e-5, 411, 0.05)
    inp = make_xattn_inputs(cfg)
    inp["Wq"] = np.zeros_like(inp["Wq"])
    inp["bq"] = np.float32(2e3 + np.random.default_rng(1).uniform(0, 1, cfg.d_q)).astype(np.float64)
    inp["Wk"], inp["bk"], inp["bv"] = np.eye(64), np.zeros(64), np.zeros(64)
    inp["M"] = np.float32(inp["M"] * 1e-3).astype(np.float64)
    inp["M"][0, 77] = np.float32(-2.9e38 + 1e35 * np.arange(64)).astype(np.float64)
    inp["Wv"] = np.float32(np.eye(64) * 1e-6).astype(np.float64)
    names = ("A", "LSE", "dQ", "dK", "dV")
    got, want = (outputs(cfg, inp, path, names) for path in (0, 1))
    for n in names:
        assert np.isfinite(want[n]).all() and np.isfinite(got[n]).all(), n
        assert off(got[n], want[n]) <= 1e-5, n


def test_products_of_small_and_large_operands():
    # values of 1e-36 have all their 24 bits in fp32, and their products with 1e30 are ordinary numbers
    cfg = XattnConfig("fr2", 1, 70, 150, 128, 192, 4, 2, 32, "fp32", "layernorm", False, False, 1e-5, 412, 0.05)
    inp = make_xattn_inputs(cfg)
    inp["M"] = np.float32(inp["M"] * 1e-36).astype(np.float64)
    inp["Wk"] = np.float32(inp["Wk"] * 1e30).astype(np.float64)
    got, ffma = (outputs(cfg, inp, path, ("K", "V", "A")) for path in (0, 1))
    exact = {"K": inp["M"] @ inp["Wk"], "V": inp["M"] @ inp["Wv"]}
    for n, want in exact.items():
        assert off(got[n], want) <= max(off(ffma[n], want), 1e-7), (n, off(got[n], want), off(ffma[n], want))
    assert off(got["A"], ffma["A"]) <= 1e-6, off(got["A"], ffma["A"])


@pytest.mark.parametrize("head_dim", [32, 64])
def test_gradients_of_a_small_output_gradient(head_dim):
    # they are linear in it; powers of two are exact, but for what fp32 itself loses of dS below 1e-38
    cfg = LayerConfig("fr3", 2, 150, 128, 128 // head_dim, 64 // head_dim, head_dim, "fp32", "layernorm", True, False, False, 1e-5, 413, 0.1)
    inp, names, small = make_inputs(cfg, affine_noise=True), ("dA", "dV", "dQ", "dK", "dWo", "dWv", "dX"), 2.0 ** -114
    away = {}
    for path in (0, 1):
        plain = outputs(cfg, inp, path, names)
        got = outputs(cfg, dict(inp, dY=inp["dY"] * small), path, names)
        away[path] = {n: off(got[n] / small, plain[n]) for n in names}
    for n in names:
        assert away[0][n] <= 2 * away[1][n] + 2e-7, (n, away[0][n], away[1][n])


@pytest.mark.parametrize("head_dim", [32, 64])
def test_gradients_under_a_small_softmax_scale(head_dim):
    # scores are all but zero at scales this small, and dQ and dK linear in them: two of the same 24 bits, powers of two apart
    names, away, bits = ("A", "dV", "dQ", "dK"), {}, float(np.float32(1.1))
    for path in (0, 1):
        runs = []
        for scale in (bits * 2.0 ** -60, bits * 2.0 ** -105):
            cfg = LayerConfig("fr10", 2, 150, 128, 128 // head_dim, 64 // head_dim, head_dim, "fp32", "layernorm", True, True, False, 1e-5, 416, 0.1, scale)
            runs.append(outputs(cfg, make_inputs(cfg, affine_noise=True), path, names))
        away[path] = {n: off(runs[1][n] * (2.0 ** 45 if n in ("dQ", "dK") else 1.0), runs[0][n]) for n in names}
    for n in names:
        assert away[0][n] <= 2 * away[1][n] + 2e-7, (n, away[0][n], away[1][n])


def test_exact_results_stay_exact():
    # the operand itself where the other one is an identity or has one entry a row, sums of integers of either sign, and the first
    # token under a causal mask, whose output is its own V
    rng = np.random.default_rng(5)
    cfg = XattnConfig("fr4", 1, 70, 192, 128, 192, 3, 3, 64, "fp32", "layernorm", False, False, 1e-5, 414, 0.05)
    inp = make_xattn_inputs(cfg)
    inp["Wk"] = np.eye(192)
    inp["Wv"] = rng.integers(-900, 900, (192, 192)).astype(np.float64)
    got = outputs(cfg, inp, 0, ("K",))
    assert np.array_equal(got["K"], inp["M"])
    inp = make_xattn_inputs(cfg)
    inp["M"] = rng.integers(-3, 90, (1, 192, 192)).astype(np.float64)
    inp["Wk"] = rng.integers(-900, 900, (192, 192)).astype(np.float64)
    got = outputs(cfg, inp, 0, ("K",))
    assert np.abs(inp["M"] @ inp["Wk"]).max() < 2 ** 24 and np.array_equal(got["K"], inp["M"] @ inp["Wk"])
    inp["M"] = np.eye(192)[None, ::-1]
    inp["Wv"] = np.float32(rng.standard_normal((192, 192)) * 10.0 ** rng.integers(-20, 20, (192, 192))).astype(np.float64)
    got = outputs(cfg, inp, 0, ("V",))
    assert np.array_equal(got["V"], inp["M"] @ inp["Wv"])
    for head_dim in (32, 64):
        cfg = LayerConfig("fr5", 2, 150, 128, 128 // head_dim, 64 // head_dim, head_dim, "fp32", "layernorm", True, True, False, 1e-5, 415, 0.1)
        got = outputs(cfg, make_inputs(cfg, affine_noise=True), 0, ("A", "V"))
        V = got["V"].reshape(2, 150, cfg.n_kv_heads, 1, head_dim).repeat(cfg.group, 3).reshape(2, 150, 128)
        assert np.array_equal(got["A"][:, 0], V[:, 0])


@pytest.mark.parametrize("cfg", [
    LayerConfig("fr6", 2, 300, 256, 4, 4, 64, "fp32", "layernorm", False, True, False, 1e-5, 421, 0.05),
    LayerConfig("fr7", 1, 700, 128, 4, 1, 32, "fp32", "rmsnorm", True, False, True, 1e-5, 422, 0.2),
    LayerConfig("fr8", 3, 190, 192, 6, 2, 64, "fp32", "layernorm", True, True, True, 1e-5, 423, 0.3),
    XattnConfig("fr9", 2, 130, 400, 128, 192, 4, 2, 32, "fp32", "rmsnorm", False, False, 1e-5, 424, 0.1),
], ids=lambda c: c.name)
def test_attention_is_no_further_off_than_multiply_adds(cfg):
    # against 64 bits, the same inputs through both kernel families; 0.2 to 0.95 of it measured
    from oracle import layer, xattn
    cross = isinstance(cfg, XattnConfig)
    inp = (make_xattn_inputs if cross else make_inputs)(cfg, affine_noise=True)
    Y, saved, grads = (xattn.xattn_fwd_bwd if cross else layer.layer_fwd_bwd)(cfg, inp)
    want = dict(grads, Y=Y, A=saved["A"])
    names = ("A", "Y", "dQ", "dK", "dV", "dX", "dWo", "dWv", "dWq", "dWk")
    got, ffma = (outputs(cfg, inp, path, names) for path in (0, 1))
    print({n: round(off(got[n], want[n]) / off(ffma[n], want[n]), 2) for n in names})
    for n in names:
        assert off(got[n], want[n]) <= off(ffma[n], want[n]), (n, off(got[n], want[n]), off(ffma[n], want[n]))
