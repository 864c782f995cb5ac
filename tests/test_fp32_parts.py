"""The parts of a split batch in the FP32 weight gradients: the scratch that a context
allocates holds those of every batch up to max_batch, they cover the batch, and they
follow from the sizes and the device alone."""
import ctypes
import random

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2106_13308_gb300 import build
    L = ctypes.CDLL(build.build())
    parts, floats = L._ZN4vqmc15gemm_simt_partsEiiiiPi, L._ZN4vqmc21gemm_simt_part_floatsEiiii
    parts.restype, parts.argtypes = ctypes.c_int, [ctypes.c_int] * 4 + [ctypes.POINTER(ctypes.c_int)]
    floats.restype, floats.argtypes = ctypes.c_size_t, [ctypes.c_int] * 4
    return parts, floats


def test_scratch_holds_every_batch(lib):
    parts, floats = lib
    rng, kpart, split = random.Random(1), ctypes.c_int(), 0
    for _ in range(1500):
        M, N, top = (int(2 ** rng.uniform(0, hi)) for hi in (12, 12, 15))
        sms = rng.choice([152, 152, 148, 16, 1])
        cap = floats(M, N, top, sms)
        assert cap <= 4 * sms * 64 * 64
        for K in [*range(1, min(top, 200)), *(rng.randint(1, top) for _ in range(40)), top]:
            p = parts(M, N, K, sms, ctypes.byref(kpart))
            assert 1 <= p <= 64
            if p > 1:
                split += 1
                assert p * M * N <= cap, (M, N, K, top, sms)
                assert kpart.value % 16 == 0 and (p - 1) * kpart.value < K <= p * kpart.value
    assert split > 1000


@pytest.mark.parametrize("M,N,K,want", [(301, 203, 777, 10), (20, 40, 1024, 16), (20, 40, 1030, 13), (65, 63, 129, 2),
                                        (20, 40, 127, 1), (64, 300, 8192, 64), (10000, 2000, 2048, 1)])
def test_number_of_parts(lib, M, N, K, want):
    assert lib[0](M, N, K, 152, ctypes.byref(ctypes.c_int())) == want
