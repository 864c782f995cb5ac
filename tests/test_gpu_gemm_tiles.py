"""The FP32 GEMMs at the sizes that choose each of their tiles (128 x 128, 64 x
128, 64 x 64 with a split batch) and at the tiles' edges, against the FP64
oracle: log pi within 1e-5 relative, the gradient within 1e-4 (the tolerances of
tests/test_gpu_parity.py), entries outside the masks exactly zero.  Each model
then takes a smaller batch: nothing of the larger one may show in it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import build_lib, er_instance, logp_rel, make_model, masked, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()
    assert torch.cuda.is_available()


CASES = [
    # n, h, B, act
    (65, 63, 129, "relu"),      # 64 x 64, one row and one sample past a tile, the batch split in two parts
    (20, 40, 1030, "sigmoid"),  # one tile, 16 parts, a ragged last part
    (130, 1900, 1025, "relu"),  # 64 x 128 for the hidden layer
    (2500, 70, 3001, "relu"),   # 128 x 128 for the output layer and its adjoint
]


@pytest.mark.parametrize("n,h,B,act", CASES)
def test_fp32_gemm_tiles_match_oracle(n, h, B, act):
    theta = inputs.lively_params(n, h, 5)
    m = make_model(n, h, B, er_instance(n, 2.0 / n, 6), act=act, theta=theta)
    P = oracle_params(theta, n, h, "fp32")
    code = oracle.RELU if act == "relu" else oracle.SIGMOID
    outside = masked(np.ones_like(theta), n, h) == 0
    for size, seed in ((B, 7), (min(B, 37), 8)):
        S = inputs.spins(size, n, seed)
        c = np.random.default_rng(seed).standard_normal(size).astype(np.float32)
        Sd = torch.from_numpy(S).cuda()
        assert logp_rel(m.logprob(Sd).cpu().numpy(), oracle.logprob(P, S, code)) <= 1e-5
        g = m.logprob_backward(Sd, torch.from_numpy(c).cuda()).cpu().numpy()
        assert rel_err(g, oracle.made_to_theta(*oracle.logprob_grad(P, S, c.astype(np.float64), code))) <= 1e-4
        assert np.all(g[outside] == 0)
    assert m.check() == 0
