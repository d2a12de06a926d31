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
