"""bench.py's account of a step: which kernels it launches and what work each is charged with (host arithmetic, no GPU)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from paper_2602_06183_b200 import binding, synth  # noqa: E402


def _account(T, D, F, V, M, flags=0, **_):
    plan = binding.sf_ffn_step_plan(binding.make_desc(T, D, F, V, M, flags=flags))
    path, held = bench._step_kernels(plan, M, flags)
    return path, held, bench._step_products(held, M)


@pytest.mark.parametrize("name", ["c1_small", "c4_d4096", "c4_d4096_m16", "c5_d8192"])
def test_every_product_is_charged_once(name):
    cfg = {k: synth.FFN_CONFIGS[name][k] for k in ("T", "D", "F", "V", "M")}
    _, held, products = _account(**cfg)
    intervals = [i for v in held.values() for i in v]
    assert len(intervals) == len(set(intervals)) and set(intervals) <= set(filter(None, bench.TRACE_NAMES))
    M = cfg["M"]
    assert sum(w for w, _ in products.values()) == 1 + 1 + 2 * 4.0 / M + 2        # y1, dy1, y3 and dX, the weight gradients


def test_weight_gradients_that_share_a_launch_are_one_entry():
    small = dict(T=1024, D=256, F=1024, V=64, M=8)
    _, held, products = _account(**small)
    assert held["gemm_dW2_dW1"] == ["gemm_dW2", "gemm_dW1"] and products["gemm_dW2_dW1"] == (2.0, 1.0)
    assert "gemm_dW1" not in held and len(held) == 7                              # the step's launches
    _, held, products = _account(T=8192, D=4096, F=16384, V=64, M=8)
    assert held["gemm_dW1"] == ["gemm_dW1"] and "gemm_dW2_dW1" not in products and len(held) == 8


def test_launches_follow_the_flags():
    m16 = dict(T=1024, D=256, F=4096, V=128, M=16)
    assert "transpose_W2" in _account(**m16)[1]
    assert "transpose_W2" not in _account(**m16, flags=binding.SF_FFN_W2_FD)[1]
    m8 = dict(T=1024, D=256, F=1024, V=64, M=8)
    assert _account(**m8)[0] == "fused" and "vnm_sparsify" not in _account(**m8)[1]
    path, held, _ = _account(**m8, flags=binding.SF_FFN_UNFUSED_ACT)
    assert path == "two_kernel" and "vnm_sparsify" in held
    assert _account(T=1024, D=256, F=1024, V=64, M=4)[0] == "plain24"


def test_measured_traffic_is_printed_for_the_captured_step_only():
    """A capture says nothing about another workload, prune mode or flags."""
    t = bench._traffic("c4_d4096", 0, 0)
    assert set(t["kernels"]) >= {"prune24_W1", "gemm_y1", "gemm_y3", "prune24_W2", "gemm_dy1", "gemm_dX", "gemm_dW2", "gemm_dW1"}
    for other in (("c5_d8192", 0, 0), ("c4_d4096", 1, 0), ("c4_d4096", 0, binding.SF_FFN_W2_FD)):
        assert bench._traffic(*other) == {}
