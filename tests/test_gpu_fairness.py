"""Small calls on one stream beside a row of large calls on another: a call of
512 MiB or more does not let the next one take the places that it leaves, so
that a small call waits for a part of one kernel at most."""
import time

import pytest

from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_small_calls_beside_a_row_of_large_ones(cuda_lib):
    T = cuda_lib
    ks = T.KeySchedule.from_triple(synth.key_triple(5))
    x = torch.zeros(1 << 30, dtype=torch.uint8, device="cuda")
    y, a = torch.empty_like(x), torch.zeros(2048, dtype=torch.uint8, device="cuda")
    b = torch.empty_like(a)
    large, small = torch.cuda.Stream(), torch.cuda.Stream()
    T.tdes_ecb_encrypt(ks, x, y, stream=large)
    T.tdes_ecb_encrypt(ks, a, b, stream=small)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    T.tdes_ecb_encrypt(ks, x, y, stream=large)
    large.synchronize()
    one = time.perf_counter() - t0
    longest = []
    for _ in range(5):
        torch.cuda.synchronize()
        for _ in range(3):
            T.tdes_ecb_encrypt(ks, x, y, stream=large)
        time.sleep(one / 5)
        waits = []
        while not large.query():
            t0 = time.perf_counter()
            T.tdes_ecb_encrypt(ks, a, b, stream=small)
            small.synchronize()
            waits.append(time.perf_counter() - t0)
        longest.append(max(waits))
    # a kernel's first CTAs end after half its time; where the next call takes their
    # places, the longest wait is 1.3 times a kernel's time
    assert sorted(longest)[2] < 0.8 * one, (longest, one)
