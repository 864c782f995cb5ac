"""The BF16 model's off-diagonal TIM energy takes the faster of its two forms: the
one kernel, or rows through memory and the general GEMM, each at sizes where the
other one is the slower (the ratio of their times on a GB300 beside them)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import act_code, make_model, oracle_params

CASES = [
    # n, h, B, act, one kernel
    (3, 40, 67, "relu", True),
    (15, 20, 70, "sigmoid", True),
    (62, 128, 40, "sigmoid", True),    # two CTAs on an SM
    (200, 300, 40, "sigmoid", True),   # one CTA on an SM
    (500, 300, 11, "sigmoid", True),
    (260, 640, 3, "relu", True),
    (2, 100, 9, "relu", False),        # 1.1
    (8, 300, 130, "sigmoid", False),   # 1.2
    (33, 200, 150, "sigmoid", False),  # 1.1
    (64, 640, 33, "sigmoid", False),   # 1.4
    (156, 500, 5, "sigmoid", False),   # 1.2
    (40, 641, 5, "relu", False),       # beyond the operand's shared memory
]
MORE = [
    # in earnest: h = 5 ln(n)^2
    (20, 44, 1024, "relu", True), (20, 44, 64, "sigmoid", True), (64, 86, 512, "sigmoid", True),
    (500, 193, 1024, "relu", True), (500, 193, 64, "sigmoid", True),
    (64, 640, 1024, "sigmoid", False), (8, 640, 128, "sigmoid", False), (1, 10, 1024, "relu", False),
]


@pytest.fixture(scope="module")
def applies():
    from paper_2106_13308_gb300 import build
    from paper_2106_13308_gb300.vqmc import ACT, PREC
    f = ctypes.CDLL(build.build())._ZN4vqmc14tim_tc_appliesEiiiiii  # vqmc::tim_tc_applies
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 6
    return lambda n, h, B, act, sms: f(PREC["bf16"], ACT[act], n, (h + 63) // 64 * 64, B, sms)


@pytest.mark.parametrize("n,h,B,act,fused", CASES + MORE)
def test_the_faster_form(applies, n, h, B, act, fused):
    assert applies(n, h, B, act, 152) == fused


@pytest.mark.gpu
@pytest.mark.parametrize("n,h,B,act,fused", CASES)
def test_energy_of_either_form(applies, n, h, B, act, fused):
    """Bounds of tests/test_gpu_tim_tiles.py; in a context of a larger max_batch the same bits."""
    assert applies(n, h, B, act, torch.cuda.get_device_properties(0).multi_processor_count) == fused
    inst = inputs.tim(n, 900 + n)
    theta = inputs.lively_params(n, h, 901 + n)
    S = inputs.spins(B, n, 902 + n)
    P = oracle_params(theta, n, h, "bf16")
    Ed = oracle.energy(inst, S)
    Eo = oracle.energy_tim_offdiag(P, S, inst["alpha"], act_code(act, "bf16"))
    J = np.abs(np.asarray(inst["J"], np.float64)).max()
    first = None
    for max_batch in (B, 3 * B + 500):
        m = make_model(n, h, max_batch, inst, act=act, precision="bf16", theta=theta)
        E = m.local_energy(torch.from_numpy(S).cuda())
        assert m.check() == 0
        e = E.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(e - (Ed + Eo)) <= n * n * 2.0 ** -16 * J + 1e-4 + 1e-3 * np.abs(Eo))
        first = E if first is None else first
        assert torch.equal(first, E)
        m.close()
