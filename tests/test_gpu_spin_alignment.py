"""Spins at any address: the conversion to the GEMMs' operands reads a row in words
that it cuts the spins from, inside the array alone, and writes whole pieces of 16."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import act_code, build_lib, er_instance, make_model, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("n,B", [(2, 1), (3, 70), (15, 5), (16, 64), (17, 65), (63, 3), (64, 66), (77, 130), (301, 9)])
def test_rows_of_any_alignment(n, B, prec):
    """log pi and the gradient from spins that start 0 to 17 bytes into a buffer filled with other values: bit for
    bit those of the same spins at the start of one, which the FP64 oracle confirms."""
    h = 20
    theta = inputs.lively_params(n, h, 5)
    m = make_model(n, h, B, er_instance(n, 1.0, 6), act="relu", precision=prec, theta=theta)
    S = inputs.spins(B, n, 7)
    c = np.random.default_rng(8).standard_normal(B).astype(np.float32)
    w = torch.from_numpy(c).cuda()
    first = torch.from_numpy(S).cuda()
    lp, g = m.logprob(first), m.logprob_backward(first, w)
    want = oracle.logprob(oracle_params(theta, n, h, prec), S, act_code("relu", prec))
    assert rel_err(lp.cpu().numpy(), want) <= (1e-5 if prec == "fp32" else 2e-3)
    for at in (1, 2, 3, 4, 7, 13, 16, 17):
        buf = torch.full((B * n + at,), 99, dtype=torch.int8, device="cuda")
        buf[at:] = first.view(-1)
        s = buf[at:].view(B, n)
        assert torch.equal(m.logprob(s).view(torch.int32), lp.view(torch.int32))
        assert torch.equal(m.logprob_backward(s, w).view(torch.int32), g.view(torch.int32))
    assert m.check() == 0
