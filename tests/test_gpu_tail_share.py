"""Tails after one step of tiles around the numbers of blocks at which a CTA's
share takes one more warp, whole and ragged: every block against the oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NCPU = max(1, min(16, os.cpu_count() or 1))


# blocks for each CTA (two on each SM), and a few more or fewer in all
@pytest.mark.parametrize("mode", ["ecb_enc", "ecb_dec", "ctr", "cbc_dec"])
@pytest.mark.parametrize("per_cta,more", [(128, 0), (128, 1), (160, 3), (192, 1), (224, 0), (224, 1), (300, 77),
                                          (384, 1), (431, -5)], ids=str)
def test_shares(cuda_lib, per_cta, more, mode):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 4 * sms * 1024 + 2 * sms * per_cta + more
    keys, iv, nonce, ctr0 = synth.key_triple(n), synth.iv64(n), synth.nonce32(n), 2**32 - n
    data = synth.random_bytes(n, 8 * n)
    ks = cuda_lib.KeySchedule.from_triple(keys)
    x = torch.from_numpy(data).cuda()
    y = torch.zeros_like(x)
    if mode == "ctr":
        cuda_lib.tdes_ctr_crypt(ks, nonce, ctr0, x, y)
        want = oracle.tdes_parallel(keys, data, "ctr", nonce=nonce, ctr0=ctr0, threads=NCPU)
    elif mode == "cbc_dec":
        cuda_lib.tdes_cbc_decrypt(ks, iv, x, y)
        d = oracle.tdes_parallel(keys, data, "ecb_dec", threads=NCPU).view(np.uint64)
        prev = np.concatenate([np.array([iv], dtype=">u8").view(np.uint64), data.view(np.uint64)[:-1]])
        want = (d ^ prev).view(np.uint8)
    else:
        call = cuda_lib.tdes_ecb_encrypt if mode == "ecb_enc" else cuda_lib.tdes_ecb_decrypt
        call(ks, x, y)
        want = oracle.tdes_parallel(keys, data, mode, threads=NCPU)
    assert np.array_equal(y.cpu().numpy(), want)
    ks.free()
