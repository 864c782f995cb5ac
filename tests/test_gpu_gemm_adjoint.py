"""The 128 x 128 tile of the FP32 hidden adjoint and of the hidden GEMM: their
epilogues, column partials (db1) and the transposed stores that the Gram kernel
reads.  Three tiles per SM are the line: small n, many units and samples."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import build_lib, er_instance, grad_blocks, make_model, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("n,h,B,act", [(70, 2500, 3001, "relu"), (33, 2497, 3100, "sigmoid")])
def test_adjoint_of_many_units(n, h, B, act):
    """The gradient within 1e-4 of the FP64 oracle in each block of parameters (tests/test_gpu_parity.py); the Gram
    matrix of the first 64 samples bit for bit that of a batch of these alone (64 x 64 tiles): every output is one
    chain over K in both."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-B // 128) * -(-h // 128) >= 3 * sms > 64 // 64 * -(-h // 64)
    theta = inputs.lively_params(n, h, 5)
    m = make_model(n, h, B, er_instance(n, 3.0 / n, 6), act=act, theta=theta)
    S = inputs.spins(B, n, 7)
    c = np.random.default_rng(8).standard_normal(B).astype(np.float32)
    Sd = torch.from_numpy(S).cuda()
    g = grad_blocks(m.logprob_backward(Sd, torch.from_numpy(c).cuda()).cpu().numpy(), n, h)
    want = grad_blocks(oracle.made_to_theta(*oracle.logprob_grad(oracle_params(theta, n, h, "fp32"), S, c.astype(np.float64),
                                                                 oracle.RELU if act == "relu" else oracle.SIGMOID)), n, h)
    for name in g:
        assert rel_err(g[name], want[name]) <= 1e-4, name
    gram = m.sr_gram(Sd)
    assert torch.equal(gram[:64, :64].contiguous().view(torch.int32), m.sr_gram(Sd[:64]).view(torch.int32))
    assert m.check() == 0
