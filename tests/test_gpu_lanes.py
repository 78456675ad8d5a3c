"""tdes_lanes_kernel (one block per thread, a table copy per lane) against the
oracle at the edges of its range: the smallest call that takes it and the
largest that does not, one to three CTAs per SM, calls of more than one wave,
every mode, both directions, EDE3 and single DES, 8-byte-aligned buffers."""
import os

import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NCPU = max(1, min(16, os.cpu_count() or 1))


def _sizes():
    return [28672, 28673, "512", "512+1", "1024", "1024+1", 196608, 300001]


def _blocks(n):
    if isinstance(n, int):
        return n
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms * int(n.split("+")[0]) + (1 if "+" in n else 0)


@pytest.mark.parametrize("mode", ["ecb_enc", "ecb_dec", "ctr", "cbc_dec"])
@pytest.mark.parametrize("size", _sizes())
def test_lanes_edges(cuda_lib, size, mode):
    n = _blocks(size)
    keys, iv = synth.key_triple(n), synth.iv64(n)
    data = synth.random_bytes(n, 8 * n)
    ks = cuda_lib.KeySchedule.from_triple(keys)
    pad = torch.empty(8 * n + 8, dtype=torch.uint8, device="cuda")
    x = pad[8:] if n % 2 else pad[:8 * n]
    x.copy_(torch.from_numpy(data))
    y = torch.zeros_like(x)
    nonce, ctr0 = synth.nonce32(n), 2**32 - n  # the last counters of the range
    with cuda_lib.small_cutoff(1 << 40):
        if mode == "ctr":
            cuda_lib.tdes_ctr_crypt(ks, nonce, ctr0, x, x)  # in place
            y = x
            want = oracle.tdes_parallel(keys, data, "ctr", nonce=nonce, ctr0=ctr0, threads=NCPU)
        elif mode == "cbc_dec":
            cuda_lib.tdes_cbc_decrypt(ks, iv, x, y)
            # D(C_i) from the oracle's ECB decryption, XORed with C_{i-1}
            d = oracle.tdes_parallel(keys, data, "ecb_dec", threads=NCPU).view(np.uint64)
            prev = np.concatenate([np.array([iv], dtype=">u8").view(np.uint64),
                                   data.view(np.uint64)[:-1]])
            want = (d ^ prev).view(np.uint8)
        else:
            call = cuda_lib.tdes_ecb_encrypt if mode == "ecb_enc" else cuda_lib.tdes_ecb_decrypt
            call(ks, x, y)
            want = oracle.tdes_parallel(keys, data, mode, threads=NCPU)
    assert np.array_equal(y.cpu().numpy(), want)
    ks.free()


def test_lanes_single_des(cuda_lib):
    n = 40001
    key = synth.key_triple(n)[:8]
    data = synth.random_bytes(n, 8 * n)
    ks = cuda_lib.KeySchedule.des(key)
    x = torch.from_numpy(data).cuda()
    with cuda_lib.small_cutoff(1 << 40):
        c = cuda_lib.tdes_ecb_encrypt(ks, x)
        assert np.array_equal(c.cpu().numpy(), oracle.des_ecb(key, data))
        assert np.array_equal(cuda_lib.tdes_ecb_decrypt(ks, c).cpu().numpy(), data)
    ks.free()
