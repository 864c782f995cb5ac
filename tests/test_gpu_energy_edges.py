"""The dense energy's field term (32 samples per CTA, sign words of 32 spins, 2048
spins at a time), the statistics of float energies (1024 per round of the CTA)
and the spins' conversion (64 x 64 tiles, 16 spins per thread) at their edges."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import act_code, build_lib, make_model, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("n,B", [(1, 1), (31, 33), (32, 32), (33, 31), (65, 64), (2048, 3), (2049, 2), (2111, 35)])
def test_dense_field_term(n, B):
    """FP32, zero couplings but for the field: E_b = sum_i h_i s_i, n FP32 additions in order."""
    rng = np.random.default_rng(40 + n)
    inst = {"kind": "dense", "n": n, "J": np.zeros((n, n), np.float32),
            "field": rng.uniform(-1, 1, n).astype(np.float32)}
    S = inputs.spins(B, n, 41 + n)
    m = make_model(n, 3, B, inst, act="relu", precision="fp32")
    E = m.local_energy(torch.from_numpy(S).cuda()).cpu().numpy()
    want = np.zeros(B, np.float32)
    for i in range(n):
        want = want + np.where(S[:, i] > 0, inst["field"][i], -inst["field"][i]).astype(np.float32)
    assert np.array_equal(E, want)


@pytest.mark.parametrize("B", [1, 31, 1023, 1024, 1025, 3000])
def test_float_statistics(B):
    """FP64 sums of float energies: 1e-12 relative, the extremes exact, the coefficients their FP32 rounding."""
    E = (np.random.default_rng(B).standard_normal(B) * 3 - 700).astype(np.float32)
    inst = {"kind": "dense", "n": 2, "J": np.zeros((2, 2), np.float32), "field": None}
    m = make_model(2, 2, B, inst, act="relu", precision="fp32")
    st, coef = m.energy_stats(torch.from_numpy(E).cuda())
    st, coef, x = st.cpu().numpy(), coef.cpu().numpy(), E.astype(np.float64)
    assert abs(st[0] - x.mean()) <= 1e-12 * abs(x.mean())
    assert abs(st[1] - x.var()) <= 1e-12 * max(x.var(), 1e-6 * x.mean() ** 2)
    assert st[2] == x.min() and st[3] == x.max()
    assert np.all(np.abs(coef - (x - x.mean()) / B) <= 2.0 ** -23 * np.abs((x - x.mean()) / B) + 1e-12 * abs(x.mean()) / B)


@pytest.mark.parametrize("n,h,B", [(63, 20, 65), (64, 130, 127), (65, 129, 128), (48, 200, 129), (130, 70, 193),
                                   (140, 64, 320), (2500, 1000, 1100)])
def test_bf16_gradient_at_tile_and_chunk_edges(n, h, B):
    """One or two K chunks of 64 per copy (K: spins, units and samples; the last case has more tiles than SMs):
    3e-2, the bound of BF16 operands."""
    theta = inputs.lively_params(n, h, 51)
    e = inputs.erdos_renyi(n, min(1.0, 4.0 / n), 52)
    m = make_model(n, h, B, inputs.to_csr(n, e, np.ones(len(e), np.int32)), act="relu", precision="bf16", theta=theta)
    S = inputs.spins(B, n, 53)
    c = np.random.default_rng(54).standard_normal(B).astype(np.float32)
    g = m.logprob_backward(torch.from_numpy(S).cuda(), torch.from_numpy(c).cuda()).cpu().numpy()
    P = oracle_params(theta, n, h, "bf16")
    want = oracle.made_to_theta(*oracle.logprob_grad(P, S, c.astype(np.float64), act_code("relu", "bf16")))
    assert rel_err(g, want) <= 3e-2
    assert m.check() == 0
