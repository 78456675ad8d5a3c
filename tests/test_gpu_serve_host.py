"""Batches of requests in pinned host memory alone run on a narrow grid; with
CBC-encryption chains, device requests beside them or staging they run on the
wide one.  Either way every result equals the oracle."""
import numpy as np
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _oracle(mode, keys, iv, data):
    if mode == 0:
        return oracle.tdes_ecb(keys, data)
    if mode == 2:
        return oracle.tdes_ctr(keys, iv >> 32, iv & 0xFFFFFFFF, data)
    return (oracle.tdes_cbc_encrypt if mode == 4 else oracle.tdes_cbc_decrypt)(keys, iv, data)


@pytest.mark.parametrize("warps", [1, 4, 8])
@pytest.mark.parametrize("what", ["host", "chains", "device_beside", "one_block"])
def test_host_requests_in_one_group(cuda_lib, what, warps):
    T = cuda_lib
    keys = synth.key_triples(41, 16)
    kt = T.KeyTable(keys)
    srv = T.Server(kt, warps_per_cta=warps)
    # more tiles than four warps on each SM take at once; ragged; a single block
    blocks = [1] if what == "one_block" else [1, 31, 33, 1025, 24 * 1024 + 7, 700001, 512, 64]
    modes = [0, 2, 3] + ([4] if what == "chains" else [])
    entries, wants = [], []
    for i, nb in enumerate(blocks * len(modes)):
        mode = modes[i // len(blocks)]
        nb = min(nb, 600) if mode == 4 else nb
        data = synth.random_bytes(4100 + i, 8 * nb)
        iv = int(synth.words(41, i, 1, synth.STREAM_IV)[0]) & 0xFFFFFFFF00000000
        x = torch.from_numpy(data)
        x = x.cuda() if what == "device_beside" and i % 5 == 0 else x.pin_memory()
        y = torch.empty_like(x) if x.is_cuda else torch.empty_like(x).pin_memory()
        entries.append((mode, i % 16, iv, x, y, 8 * nb))
        wants.append((mode, keys[i % 16].tobytes(), iv, data))
    torch.cuda.synchronize()
    assert srv.wait_group(srv.submit_group(entries), 60.0) == 0
    for e, w in zip(entries, wants):
        assert (e[4].cpu().numpy() == _oracle(*w)).all(), (e[0], e[5])
    srv.close()
