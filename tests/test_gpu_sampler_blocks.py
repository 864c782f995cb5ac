"""The blocked CUDA-core sampler at the edges of its blocks (16 steps), unit
groups (16), chunks (64 units), 8 samples per CTA and 128 units per warp and
round, against the FP64 oracle on shared uniforms.  Tolerances as for every
sampler (tests/test_gpu_parity.py): each draw with |u - p_i| >= 1e-6 equals
[u < p_i] of the oracle's conditional on the sample's own prefix (BF16: except
where an ambiguous hidden unit can move the logit across), log pi within 1e-5
relative."""
import pytest
import torch

from paper_2106_13308_gb300 import inputs

from gpu_helpers import (act_code, bf16_sample_check, build_lib, er_instance, logp_rel, make_model, oracle_params,
                         rows_without_near_ties, teacher_forced)

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()
    assert torch.cuda.is_available()


CASES = [
    # n, h, B, act, precision, sampler
    (1, 3, 1, "relu", "fp32", "cuda_core"),       # no unit completes before the only step
    (17, 16, 8, "sigmoid", "bf16", "cuda_core"),  # one group, its last unit complete at the last step
    (18, 17, 9, "relu", "fp32", "cuda_core"),     # the second group has one unit
    (64, 64, 7, "relu", "bf16", "cuda_core"),     # hp = h = 64
    (33, 65, 5, "sigmoid", "fp32", "cuda_core"),  # two units a step, hp = 128
    (5, 300, 3, "relu", "bf16", "cuda_core"),     # groups completed without a step of their own
    (97, 20, 17, "relu", "bf16", "cuda_core"),    # several blocks to a group, a short last one
    (144, 128, 16, "sigmoid", "bf16", "cuda_core"),   # a whole round of the 128 pair classes
    (150, 300, 4, "relu", "fp32", "cuda_core"),   # more than one round; U beyond one round of a warp
    (700, 650, 3, "relu", "bf16", "cuda_core"),   # U wraps over the four warps
    (80, 40, 11, "sigmoid", "fp32", "cuda_core_wide"),
    (300, 290, 9, "relu", "bf16", "cuda_core_wide"),
]


@pytest.mark.parametrize("n,h,B,act,prec,sampler", CASES)
def test_blocked_sampler_matches_oracle(n, h, B, act, prec, sampler):
    theta = inputs.lively_params(n, h, 3)
    m = make_model(n, h, B, er_instance(n, min(1.0, 3.0 / n), 2), act=act, precision=prec, theta=theta, sampler=sampler)
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
