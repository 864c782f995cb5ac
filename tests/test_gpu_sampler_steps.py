"""The CUDA-core sampler that goes step by step, in each of its shapes (up to 64,
1024 and 2048 hidden units, beyond, and wide): against the FP64 oracle on shared
uniforms, with the tolerances of tests/test_gpu_sampler_blocks.py, and bit for bit
against the blocked sampler, which takes another batch of the same model."""
import ctypes

import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import (act_code, bf16_sample_check, build_lib, er_instance, logp_rel, make_model, oracle_params,
                         rows_without_near_ties, teacher_forced)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stepwise():
    from paper_2106_13308_gb300.vqmc import ACT, LIB_PATH, PREC
    build_lib()
    f = ctypes.CDLL(LIB_PATH)._ZN4vqmc16sampler_stepwiseEiiiiibi  # vqmc::sampler_stepwise
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 5 + [ctypes.c_bool, ctypes.c_int]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return lambda prec, act, n, h, B, sampler: f(PREC[prec], ACT[act], n, h, B, sampler == "cuda_core_wide", sms)


@pytest.mark.parametrize("n,h,act,prec,sampler,blocked,stepped", [
    (40, 20, "relu", "bf16", "cuda_core", 1024, 20001),
    (20, 40, "sigmoid", "fp32", "cuda_core", 1024, 20001),
    (130, 700, "relu", "bf16", "cuda_core", 1300, 3001),
    (100, 900, "relu", "fp32", "cuda_core", 300, 1301),
    (150, 1100, "relu", "bf16", "cuda_core", 300, 1301),
    (500, 2500, "relu", "bf16", "cuda_core", 3000, 301),
    (130, 700, "relu", "fp32", "cuda_core_wide", 700, 9),
])
def test_both_samplers_give_the_same_bits(stepwise, n, h, act, prec, sampler, blocked, stepped):
    assert not stepwise(prec, act, n, h, blocked, sampler) and stepwise(prec, act, n, h, stepped, sampler)
    m = make_model(n, h, max(blocked, stepped), er_instance(n, 3.0 / n, 2), act=act, precision=prec,
                   theta=inputs.lively_params(n, h, 3), sampler=sampler)
    k = min(blocked, stepped)
    (s0, l0), (s1, l1) = m.sample(blocked, None, iteration=5), m.sample(stepped, None, iteration=5)
    assert torch.equal(s0[:k], s1[:k]) and torch.equal(l0[:k].view(torch.int32), l1[:k].view(torch.int32))
    assert m.check() == 0


@pytest.mark.parametrize("n,h,B,act,prec,sampler", [
    (30, 20, 20001, "relu", "fp32", "cuda_core"),  # one warp per group
    (24, 33, 9001, "sigmoid", "bf16", "cuda_core"),
    (30, 900, 3, "relu", "bf16", "cuda_core"),     # two warps; several slots of a lane complete at a step
    (40, 1024, 9, "sigmoid", "fp32", "cuda_core"),
    (33, 1500, 2, "relu", "fp32", "cuda_core"),    # four groups of two warps
    (50, 2048, 5, "sigmoid", "bf16", "cuda_core"),
    (60, 2800, 3, "relu", "fp32", "cuda_core"),    # four warps per group
    (70, 5120, 6, "relu", "bf16", "cuda_core"),
    (20, 400, 7, "sigmoid", "bf16", "cuda_core_wide"),
])
def test_stepped_sampler_matches_oracle(stepwise, n, h, B, act, prec, sampler):
    assert stepwise(prec, act, n, h, B, sampler)
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
