"""Calls whose kernels may start while the one before still runs (they stage their
tables first): chains of dependent calls on one stream, eager and in a CUDA graph,
over every kernel family, between each other and beside torch's own kernels."""
import pytest

import oracle
from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one block per thread, per-lane tables, one-warp CTAs, wide grids with and
# without a tail, ragged
SIZES = [64, 28672, 100000, 300001, 700 * 1024 + 3, 1300 * 1024]


def _chain(T, ks, kd, x, a, b, nonce, iv, n):
    """D(E(x)) by ECB, CTR twice, single DES both ways, CBC decryption of the
    ECB encryption: a ends as x, b as the CBC plaintext."""
    T.tdes_ecb_encrypt(ks, x, a)
    T.tdes_cbc_decrypt(ks, iv, a, b)
    T.tdes_ecb_decrypt(ks, a, a)
    T.tdes_ctr_crypt(ks, nonce, 7, a, a)
    T.tdes_ecb_encrypt(kd, a, a)
    T.tdes_ecb_decrypt(kd, a, a)
    a.add_(1).sub_(1)  # torch's kernels between ours
    T.tdes_ctr_crypt(ks, nonce, 7, a, a)


@pytest.mark.parametrize("graph", [False, True], ids=["stream", "graph"])
@pytest.mark.parametrize("n", SIZES)
def test_dependent_calls(cuda_lib, n, graph):
    T = cuda_lib
    keys, iv, nonce = synth.key_triple(n), synth.iv64(n), synth.nonce32(n)
    ks, kd = T.KeySchedule.from_triple(keys), T.KeySchedule.des(keys[:8])
    data = torch.from_numpy(synth.random_bytes(n, 8 * n)).cuda()
    x, a, b = data.clone(), torch.empty_like(data), torch.empty_like(data)
    cutoff = 1 << 40 if n <= 300001 else 0
    with T.small_cutoff(cutoff):
        run = lambda: _chain(T, ks, kd, x, a, b, nonce, iv, n)  # noqa: E731
        run()
        torch.cuda.synchronize()
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                run()
            run = g.replay
        for _ in range(5):
            a.zero_()
            b.zero_()
            run()
            x.copy_(a)  # the next pass reads what this one wrote
        torch.cuda.synchronize()
    assert torch.equal(x, data)
    # CBC plaintext: D(C_i) ^ C_{i-1} = x_i ^ E(x_{i-1}); a sample against the oracle
    m = min(n, 2000)
    want = oracle.tdes_cbc_decrypt(keys, iv, oracle.tdes_ecb(keys, data[:8 * m].cpu().numpy()))
    assert (b[:8 * m].cpu().numpy() == want).all()


def test_chain_encryptions_follow_each_other(cuda_lib):
    T = cuda_lib
    keys, iv = synth.key_triple(3), synth.iv64(3)
    ks = T.KeySchedule.from_triple(keys)
    data = synth.random_bytes(3, 8 * 40)
    x = torch.from_numpy(data).cuda()
    want = data
    for _ in range(6):  # in place, each reading the one before
        T.tdes_cbc_encrypt(ks, iv, x, x)
        want = oracle.tdes_cbc_encrypt(keys, iv, want)
    assert (x.cpu().numpy() == want).all()
