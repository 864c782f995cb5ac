"""FP32 contexts: the gradient of a batch depends on the batch alone, and the
context holds what its calls read."""
import numpy as np
import pytest
import torch

from paper_2106_13308_gb300 import inputs

from gpu_helpers import build_lib, er_instance, make_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


@pytest.mark.parametrize("n,h,B", [(301, 203, 777), (500, 193, 1024), (40, 700, 500), (65, 63, 129), (20, 40, 64)])
def test_gradient_bits_do_not_depend_on_max_batch(n, h, B):
    """The same parameters, samples and weights in contexts of several max_batch, the batch split into as many
    parts in each: equal bits."""
    theta = inputs.lively_params(n, h, 5)
    S = torch.from_numpy(inputs.spins(B, n, 7)).cuda()
    c = torch.from_numpy(np.random.default_rng(8).standard_normal(B).astype(np.float32)).cuda()
    grads = []
    for max_batch in (B, B + 1, 4096, 9000):
        m = make_model(n, h, max_batch, er_instance(n, 3.0 / n, 6), act="relu", theta=theta)
        grads.append(m.logprob_backward(S, c))
        assert m.check() == 0
        m.close()
    for g in grads[1:]:
        assert torch.equal(grads[0].view(torch.int32), g.view(torch.int32))


@pytest.mark.parametrize("n,h,B", [(10000, 2000, 16), (64, 2000, 16384)])
def test_context_holds_what_its_calls_read(n, h, B):
    """Device memory of a new FP32 context: parameters, moments and gradient, three copies of the weights, the
    spins in two forms, the output adjoint in two, hidden activations and their adjoint in one (their transposes
    come with the first SR call), partial sums, and 40 MB for the rest and the allocator's rounding."""
    e = inputs.erdos_renyi(n, 2.0 / n, 1)
    inst = inputs.to_csr(n, e, np.ones(len(e), np.int32))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    m = make_model(n, h, B, inst, act="relu", precision="fp32")
    used = free - torch.cuda.mem_get_info()[0]
    weights, spins, hidden = 4.0 * n * h, 4.0 * n * B, 4.0 * h * B
    assert used <= 4 * 2 * weights + 3 * weights + 4.1 * spins + 2.1 * hidden + 40e6
    S = m.sample(16, None)[0]
    E = m.local_energy(S)
    before = m.grad(S, E)[0]
    if h * n <= 2e6:
        assert m.sr_gram(S).isfinite().all()
    assert torch.equal(before, m.grad(S, E)[0]) and m.check() == 0
    m.close()
