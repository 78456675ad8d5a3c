"""What follows a uniform call or a batch on the same stream, with nothing waited
for in between, reads finished output: the calls' last kernels start beside the
ones before them, and the call that follows may start beside the last.  Each
chain is compared with the same calls with a synchronise after each."""
import numpy as np
import pytest

from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _consumers(T, dst):
    """Calls that read dst: a wide one over all of it, one CTA and a chain over its
    first, middle and last blocks."""
    ks = T.KeySchedule.from_triple(synth.key_triple(17))
    n = dst.numel()
    wide = torch.empty_like(dst)
    spots = [0, n // 16 * 8, n - 512]
    outs = [torch.empty(512, dtype=torch.uint8, device="cuda") for _ in range(2 * len(spots))]

    def run():
        for i, s in enumerate(spots):
            T.tdes_ctr_crypt(ks, 3, 0, dst[s:s + 512], outs[i])
        T.tdes_ecb_encrypt(ks, dst, wide)
        for i, s in enumerate(spots):
            T.tdes_cbc_encrypt(ks, 5, dst[s:s + 512], outs[len(spots) + i])

    return run, [wide, *outs]


def _check(T, produce, dst, graph):
    consume, outs = _consumers(T, dst)

    def both():
        produce()
        consume()

    produce()
    torch.cuda.synchronize()
    want_dst = dst.clone()
    consume()
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            both()
        both = g.replay
    for _ in range(4):
        dst.zero_()
        for o in outs:
            o.zero_()
        both()
        torch.cuda.synchronize()
        assert torch.equal(dst, want_dst)
        assert all(torch.equal(o, w) for o, w in zip(outs, want))


# (message bytes, messages): chains first; all messages in 8 CTAs' worth of
# tiles; over 64 MiB of 8- and 16-byte messages, where the chains come last
@pytest.mark.parametrize("graph", [False, True], ids=["stream", "graph"])
@pytest.mark.parametrize("msg,n,keys", [(64, 1 << 17, 4096), (200, 40001, 16), (8, 9_000_001, 1 << 12),
                                        (16, 4_500_001, 8)], ids=str)
def test_after_a_uniform_call(cuda_lib, msg, n, keys, graph):
    T = cuda_lib
    words = lambda stream: torch.from_numpy(synth.u64s(msg, n, stream).view(np.int64)).cuda()  # noqa: E731
    kt = T.KeyTable(synth.key_triples(msg, keys))
    key_index = (words(synth.STREAM_KEYPICK) & (keys - 1)).to(torch.int32)
    mode = torch.tensor([0, 2, 3, 4, 4], dtype=torch.uint8, device="cuda")[
        (words(synth.STREAM_MODE) & 0xFFFF) * 5 >> 16]
    iv = words(synth.STREAM_IV) & -(1 << 32)
    src = torch.empty(n * msg, dtype=torch.uint8, device="cuda")
    synth.fill_device(src, msg)
    dst = torch.zeros_like(src)
    need = T.tdes_uniform_scratch_bytes(kt, n, msg)
    buf = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    scratch = buf[-buf.data_ptr() % 256:][:need]
    _check(T, lambda: T.tdes_uniform_crypt(kt, key_index, mode, iv, src, dst, msg, scratch=scratch), dst,
           graph)


# mixed-key tiles that outlast a few scalar items, a few short chains, long
# chains and tiles of larger messages, and the other way round
@pytest.mark.parametrize("graph", [False, True], ids=["stream", "graph"])
@pytest.mark.parametrize("small,medium,chains,large", [(60000, 0, [5, 1, 3], 0), (0, 3000, [2], 0),
                                                       (9000, 0, [700, 400, 90], 0),
                                                       (2000, 300, [], 40)], ids=str)
def test_after_a_batch(cuda_lib, small, medium, chains, large, graph):
    T = cuda_lib
    nb = ([1 + i % 32 for i in range(small)] + [33 + 37 * i % 480 for i in range(medium)] + chains
          + [5000 + 11 * i for i in range(large)])
    modes = [4 if i >= small + medium and i < small + medium + len(chains) else (0, 2, 3, 1)[i % 4]
             for i in range(len(nb))]
    offs = np.concatenate([[0], np.cumsum(8 * np.array(nb, dtype=np.int64))])
    src = torch.empty(int(offs[-1]), dtype=torch.uint8, device="cuda")
    synth.fill_device(src, len(nb))
    dst = torch.zeros_like(src)
    kt = T.KeyTable(synth.key_triples(len(nb), 64))
    plan = T.Batch(kt, [(modes[i], i % 64, i << 32, src.data_ptr() + int(offs[i]),
                         dst.data_ptr() + int(offs[i]), 8 * nb[i]) for i in range(len(nb))])
    assert plan.info()["n_mixed_tiles"] > 0
    _check(T, plan.launch, dst, graph)
    _check(T, plan.launch_graph, dst, False)
