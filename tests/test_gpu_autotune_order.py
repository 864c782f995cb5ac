"""The batch autotuner's choice of a CUDA-core member's summation order: timed only
where the two orders are kernels of different shape, so that noise does not choose
the rounding."""
import numpy as np
import pytest
import torch

from paper_2106_13308_gb300 import inputs

from gpu_helpers import build_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()


def _problem(n, h, B, sampler):
    e = inputs.erdos_renyi(n, 3.0 / n, n)
    return dict(n=n, h=h, max_batch=B, instance=inputs.to_csr(n, e, np.ones(len(e), np.int32)), act="relu",
                precision="bf16", seed=n, sampler=sampler)


def test_blocked_members_keep_the_default_order():
    """Both orders in blocks of steps (small models, where a timing of the two differs by noise alone, and the
    batch configuration's h = n): the default one, whatever the member asked for; every member advances alike."""
    from paper_2106_13308_gb300.vqmc import VQMCBatch
    probs = [_problem(20 + q, 20 + q, 8, s) for q in range(12) for s in ("cuda_core", "cuda_core_wide")]
    probs += [_problem(300, 300, 64, s) for s in ("cuda_core", "cuda_core_wide")]
    probs.append(_problem(20, 640, 64, "cuda_core"))  # the wide order steps here, and is 1.6 times as fast
    batch = VQMCBatch(probs)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        batch.autotune([p["max_batch"] for p in probs])
        stream.synchronize()
    samplers = batch.schedule()[2]
    assert samplers[:-1] == ["cuda_core"] * (len(probs) - 1)
    assert samplers[-1] in ("cuda_core", "cuda_core_wide")
    assert len({m.iteration for m in batch.members}) == 1 and all(m.check() == 0 for m in batch.members)
    batch.close()
