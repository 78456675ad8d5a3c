"""Calls around the steps of one tile per SM sub-partition, where the last
blocks run one per thread after the tiles: just below, at and above a step, at
and past the longest tail, ragged ends, every mode; single DES and 8-byte
alignment, which keep tiles to the end."""
import os

import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NCPU = max(1, min(16, os.cpu_count() or 1))


def _blocks(steps, extra):
    return steps * 4 * torch.cuda.get_device_properties(0).multi_processor_count * 1024 + extra


# (steps, extra blocks): tails of 0, 1 block, a ragged one, the longest (128
# tiles, 320 after a whole number of passes) and one block more
SPLITS = [(1, -1), (1, 0), (1, 1), (1, 128 * 1024), (1, 128 * 1024 + 1), (2, 19 * 1024 + 517),
          (3, 77 * 1024), (4, 320 * 1024), (4, 320 * 1024 + 1)]


def _check(cuda_lib, keys, data, mode, x, y, des=False):
    n = data.size // 8
    iv, nonce, ctr0 = synth.iv64(n), synth.nonce32(n), 2**32 - n
    ks = cuda_lib.KeySchedule.des(keys[:8]) if des else cuda_lib.KeySchedule.from_triple(keys)
    k24 = keys[:8] * 3 if des else keys
    x.copy_(torch.from_numpy(data))
    if mode == "ctr":
        cuda_lib.tdes_ctr_crypt(ks, nonce, ctr0, x, y)
        want = oracle.tdes_parallel(k24, data, "ctr", nonce=nonce, ctr0=ctr0, threads=NCPU)
    elif mode == "cbc_dec":
        cuda_lib.tdes_cbc_decrypt(ks, iv, x, y)
        d = oracle.tdes_parallel(k24, data, "ecb_dec", threads=NCPU).view(np.uint64)
        prev = np.concatenate([np.array([iv], dtype=">u8").view(np.uint64), data.view(np.uint64)[:-1]])
        want = (d ^ prev).view(np.uint8)
    else:
        cuda_lib.tdes_ecb_encrypt(ks, x, y)
        want = oracle.tdes_parallel(k24, data, "ecb_enc", threads=NCPU)
    assert np.array_equal(y.cpu().numpy(), want)
    ks.free()


# the split is the same code in every mode: all edges in ECB, tails in the others
CASES = [(s, "ecb_enc") for s in SPLITS] + [(s, m) for s in SPLITS[2:6] for m in ("ctr", "cbc_dec")]


@pytest.mark.parametrize("split,mode", CASES, ids=str)
def test_tail_splits(cuda_lib, split, mode):
    """The whole output against the oracle: every block of tiles and tail."""
    n = _blocks(*split)
    x = torch.empty(8 * n, dtype=torch.uint8, device="cuda")
    _check(cuda_lib, synth.key_triple(n), synth.random_bytes(n, 8 * n), mode, x, torch.zeros_like(x))


@pytest.mark.parametrize("mode", ["ecb_enc", "ctr", "cbc_dec"])
@pytest.mark.parametrize("form", ["in_place", "offset8", "des"])
def test_tail_forms(cuda_lib, form, mode):
    n = _blocks(1, 4097)
    pad = torch.empty(8 * n + 8, dtype=torch.uint8, device="cuda")
    x = pad[8:] if form == "offset8" else pad[:8 * n]
    y = x if form == "in_place" else torch.zeros_like(pad)[8:] if form == "offset8" else torch.zeros_like(x)
    _check(cuda_lib, synth.key_triple(n), synth.random_bytes(n, 8 * n), mode, x, y, des=form == "des")
