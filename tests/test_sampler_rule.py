"""The choice between the two CUDA-core samplers (both give the same bits): in
blocks of steps where a block has steps to hold, step by step where many units
complete at a step or where a small model's batch needs many more rounds of CTAs.
Each case was measured on a GB300 (152 SMs) in both, the ratio of their times is
beside it."""
import ctypes

import pytest

SMS = 152


@pytest.fixture(scope="module")
def stepwise():
    from paper_2106_13308_gb300 import build
    from paper_2106_13308_gb300.vqmc import ACT, PREC
    f = ctypes.CDLL(build.build())._ZN4vqmc16sampler_stepwiseEiiiiibi  # vqmc::sampler_stepwise
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 5 + [ctypes.c_bool, ctypes.c_int]
    return lambda prec, act, n, h, B, wide=False: f(PREC[prec], ACT[act], n, h, B, wide, SMS)


@pytest.mark.parametrize("prec,act,n,h,B,wide", [
    ("bf16", "relu", 300, 4800, 64, False),      # 4.5 times
    ("bf16", "sigmoid", 100, 5000, 8, False),    # 4.7
    ("fp32", "relu", 300, 2400, 8, False),       # 2.1
    ("bf16", "relu", 500, 4000, 512, False),     # 2.5
    ("bf16", "relu", 64, 2000, 64, False),       # 1.9
    ("fp32", "relu", 100, 1600, 64, False),      # 1.9
    ("bf16", "relu", 100, 800, 8192, False),     # 1.4
    ("fp32", "relu", 200, 1600, 64, True),       # 1.6 and more
    ("fp32", "sigmoid", 20, 20, 8192, False),    # 1.3
    ("bf16", "relu", 1000, 50, 8192, False),     # 1.2
    ("bf16", "relu", 400, 40, 65536, False),     # 1.9
])
def test_step_by_step(stepwise, prec, act, n, h, B, wide):
    assert stepwise(prec, act, n, h, B, wide)


@pytest.mark.parametrize("prec,act,n,h,B,wide", [
    ("bf16", "relu", 1000, 1000, 4096, False),   # 0.3
    ("fp32", "relu", 10000, 2000, 2048, False),  # 0.6
    ("bf16", "relu", 2000, 2000, 8192, False),   # 0.4
    ("bf16", "relu", 5000, 5000, 512, False),    # 0.7
    ("fp32", "sigmoid", 20, 40, 1024, False),    # 0.4
    ("fp32", "relu", 500, 193, 1024, False),     # 0.2
    ("bf16", "relu", 300, 1200, 64, False),      # 0.6
    ("bf16", "relu", 64, 64, 4864, False),       # 0.5
    ("bf16", "relu", 10, 10, 8192, True),        # 0.2
    ("bf16", "relu", 200, 1600, 2048, True),     # 0.5
])
def test_in_blocks(stepwise, prec, act, n, h, B, wide):
    assert not stepwise(prec, act, n, h, B, wide)
