"""The blocked CUDA-core sampler with more than 1024 hidden units after the first
group: a warp's second round of the pre-activations' update, whose weights are
loaded 16 rows ahead in BF16 and 8 in FP32, in each of the summation orders.
Oracle and tolerances as in tests/test_gpu_sampler_blocks.py."""
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import (act_code, bf16_sample_check, build_lib, er_instance, logp_rel, make_model, oracle_params,
                         rows_without_near_ties, teacher_forced)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("n,h,B,act,prec,sampler", [
    (1300, 1200, 9, "relu", "bf16", "cuda_core"),
    (1100, 1090, 5, "relu", "fp32", "cuda_core"),
    (1250, 1201, 4, "sigmoid", "bf16", "cuda_core_wide"),
    (1200, 1130, 3, "sigmoid", "fp32", "cuda_core_wide"),
])
def test_second_round_matches_oracle(n, h, B, act, prec, sampler):
    theta = inputs.lively_params(n, h, 3)
    m = make_model(n, h, B, er_instance(n, 3.0 / n, 2), act=act, precision=prec, theta=theta, sampler=sampler)
    P = oracle_params(theta, n, h, prec)
    U = inputs.uniforms(B, n, 4)
    S, lp = m.sample(B, torch.from_numpy(U).cuda())
    S, lp = S.cpu().numpy(), lp.cpu().numpy()
    assert m.check() == 0
    code = act_code(act, prec)
    if prec == "fp32":
        mism, ties = teacher_forced(P, S, U, code)
        assert mism == 0, (mism, ties)
        So, lpo = oracle.sample(P, U, code)
        rows = rows_without_near_ties(P, So, U, code, 1e-6)
        assert (S[rows] == So[rows]).all()
        assert logp_rel(lp[rows], lpo[rows]) <= 1e-5
    else:
        c = bf16_sample_check(P, S, U, code, lp=lp)
        assert c["unflagged_mismatches"] == 0 and c["clean_rows_equal"] and c["logp_within_bound"], c
