"""The one-kernel off-diagonal TIM energy of the BF16 model at the edges of its
tiles: 31 flips of a sample per tile (several samples in a group of 32 rows
below 16 spins), 4 samples or more per tile, 128 outputs per output tile, and
hidden sizes on both sides of the two-CTA, one-CTA and general forms."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_13308_gb300 import inputs

from gpu_helpers import act_code, build_lib, make_model, oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("n,h,B,act", [
    (1, 3, 5, "relu"), (2, 1, 67, "relu"), (15, 20, 9, "sigmoid"), (16, 70, 8, "relu"), (31, 64, 7, "relu"),
    (32, 65, 3, "relu"), (62, 128, 4, "sigmoid"), (63, 40, 1, "relu"), (127, 100, 6, "relu"), (128, 130, 5, "relu"),
    (129, 257, 2, "relu"), (156, 300, 11, "sigmoid"), (260, 640, 3, "relu"), (40, 641, 5, "relu"),
])
def test_tim_energy_at_tile_edges(n, h, B, act):
    """The bounds are those of the general form: the diagonal's FP32 sums
    (n^2 terms) and 1e-3 of the off-diagonal energy (FP32 sums of log pi and a
    hidden activation that rounds the other way in one row of a pair)."""
    inst = inputs.tim(n, 900 + n)
    theta = inputs.lively_params(n, h, 901 + n)
    S = inputs.spins(B, n, 902 + n)
    m = make_model(n, h, B, inst, act=act, precision="bf16", theta=theta)
    E = m.local_energy(torch.from_numpy(S).cuda()).cpu().numpy().astype(np.float64)
    P = oracle_params(theta, n, h, "bf16")
    Ed = oracle.energy(inst, S)
    Eo = oracle.energy_tim_offdiag(P, S, inst["alpha"], act_code(act, "bf16"))
    J = np.abs(np.asarray(inst["J"], np.float64)).max()
    assert np.all(np.abs(E - (Ed + Eo)) <= n * n * 2.0 ** -16 * J + 1e-4 + 1e-3 * np.abs(Eo))
    assert m.check() == 0
