"""The scalar block rounds and the counter bit-planes the kernels take, compiled
for the host (tests/host_check/tdes_host_scalar.cu): the rounds against the
oracle, the planes against the counter blocks they stand for."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import build, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not os.path.exists(build.nvcc()) and shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hs") / "tdes_host_scalar")
    subprocess.check_call([build.nvcc(), "-O1", "-std=c++17", "-o", out,
                           os.path.join(ROOT, "tests", "host_check", "tdes_host_scalar.cu")])
    return out


def _run(*args, data=b""):
    r = subprocess.run(list(map(str, args)), input=data, capture_output=True, timeout=120)
    assert r.returncode == 0
    return r.stdout


KEYSETS = {"seeded": lambda: synth.key_triple(81),
           "single": lambda: synth.key_triple(82)[:8] * 3,
           "weak": lambda: b"\x01" * 8 + b"\xfe" * 8 + synth.key_triple(83)[:8]}


@pytest.mark.parametrize("keys", KEYSETS)
@pytest.mark.parametrize("mode", ["sw_enc", "sw_dec", "s1_enc", "s1_dec"])
def test_swap_rounds_match_oracle(exe, keys, mode):
    k = KEYSETS[keys]()
    data = np.concatenate([synth.random_bytes(84, 8 * 100),  # and every single-bit block
                           np.array([1 << i for i in range(64)], dtype=">u8").view(np.uint8)])
    got = np.frombuffer(_run(exe, mode, k.hex(), data=data.tobytes()), dtype=np.uint8)
    dec = mode.endswith("dec")
    want = (oracle.des_ecb(k[:8], data, decrypt=dec) if mode[:2] == "s1"
            else oracle.tdes_ecb(k, data, decrypt=dec))
    assert np.array_equal(got, want)


# (first counter of the tile): no carry, carries out of the slots' bits (0 and
# 6..9) and through all bits up to 31, and the last tile of the counter range
COUNTERS = [0, 1, 0x3F, 0x3C0, 0x3FF, 0xFFFF, 0x7FFFFC00, 0x7FFFFFFF, 0xFFFFFC00, 0xA5C3965A]


@pytest.mark.parametrize("c", COUNTERS, ids=hex)
def test_counter_planes_are_the_counter_blocks(exe, c):
    nonce = 0x8000F00D ^ (c * 0x9E3779B1 & 0xFFFFFFFF)
    for lane in range(32):
        got = np.frombuffer(_run(exe, "planes", nonce, c, lane), dtype="<u4").reshape(2, 32)
        # slot 2j + h: counter c + 64 j + 2 lane + h, big-endian behind the nonce
        ctr = [(c + 64 * (s // 2) + 2 * lane + s % 2) & 0xFFFFFFFF for s in range(32)]
        words = [[int.from_bytes(nonce.to_bytes(4, "big"), "little")] * 32,
                 [int.from_bytes(x.to_bytes(4, "big"), "little") for x in ctr]]
        for half in range(2):
            for k in range(32):  # plane k: bit k of every slot's word
                want = sum((words[half][s] >> k & 1) << s for s in range(32))
                assert int(got[half, k]) == want, (lane, half, k)
