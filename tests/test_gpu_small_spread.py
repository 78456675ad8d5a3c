"""Calls of 2 to 16 CTAs of 128 blocks each, whose CTAs have more threads than
blocks: around the ends of that range and of a CTA, every mode, EDE3 and single
DES, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("des", [False, True], ids=["ede3", "des"])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 1000, 1920, 1921, 2047, 2048, 2049])
def test_small_calls(cuda_lib, n, des):
    T, keys, iv, nonce, ctr0 = cuda_lib, synth.key_triple(n), synth.iv64(n), synth.nonce32(n), 2**32 - n
    data = synth.random_bytes(n, 8 * n)
    k24 = keys[:8] * 3 if des else keys
    ks = T.KeySchedule.des(keys[:8]) if des else T.KeySchedule.from_triple(keys)
    x = torch.from_numpy(data).cuda()
    y = torch.zeros(8 * n + 64, dtype=torch.uint8, device="cuda")  # and nothing past the end
    cases = [(lambda o: T.tdes_ecb_encrypt(ks, x, o), oracle.tdes_ecb(k24, data)),
             (lambda o: T.tdes_ecb_decrypt(ks, x, o), oracle.tdes_ecb(k24, data, decrypt=True)),
             (lambda o: T.tdes_ctr_crypt(ks, nonce, ctr0, x, o), oracle.tdes_ctr(k24, nonce, ctr0, data)),
             (lambda o: T.tdes_cbc_decrypt(ks, iv, x, o), oracle.tdes_cbc_decrypt(k24, iv, data))]
    for call, want in cases:
        y.zero_()
        call(y[:8 * n])
        got = y.cpu().numpy()
        assert np.array_equal(got[:8 * n], want) and not got[8 * n:].any()
    ks.free()
