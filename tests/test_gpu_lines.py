"""Where a rule takes a call to another path, the call takes no longer there than
its neighbour on the other side.  Both are timed in turn, so that whatever else
moves moves both; the limits leave 8% for the events' grain (2 us) and spread."""
import numpy as np
import pytest

from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ratio(a, b, rows=1, rounds=60):
    """Time of `rows` calls of a, out of L2, over that of b, taken in turn (means
    of the middle half)."""
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    times = ([], [])
    for i in range(rounds + 3):
        for call, out in zip((a, b), times):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            flush.zero_()
            e0.record()
            for _ in range(rows):
                call()
            e1.record()
            e1.synchronize()
            if i >= 3:
                out.append(e0.elapsed_time(e1))
    mid = [np.mean(sorted(t)[rounds // 4:-(rounds // 4)]) for t in times]
    return float(mid[0] / mid[1])


def _medium(cuda_lib, nb, blocks):
    """A plan of messages of nb blocks, `blocks` in all or the last ones fewer."""
    n = blocks // nb
    src = torch.zeros(8 * nb * n, dtype=torch.uint8, device="cuda")
    synth.fill_device(src, nb)
    dst = torch.empty_like(src)
    kt = cuda_lib.KeyTable(synth.key_triples(nb, 64))
    plan = cuda_lib.Batch(kt, [((0, 2, 3, 1)[i % 4], i % 64, i << 32, src.data_ptr() + 8 * nb * i,
                                dst.data_ptr() + 8 * nb * i, 8 * nb) for i in range(n)])
    return plan, (kt, src, dst)


@pytest.mark.parametrize("nb", [33, 48, 64, 512])
def test_medium_messages_past_the_line(cuda_lib, nb):
    """131072 blocks of medium messages as mixed-key tiles, and one message fewer
    as scalar items."""
    blocks = -(-131072 // nb) * nb
    past, hold = _medium(cuda_lib, nb, blocks)
    before, hold2 = _medium(cuda_lib, nb, blocks - nb)
    assert past.info()["n_mixed_tiles"] > 0 and before.info()["n_mixed_tiles"] == 0
    r = _ratio(past.launch_graph, before.launch_graph)
    del hold, hold2
    assert r <= 1.08, r


def _single_key(cuda_lib, mode, longest):
    """A function that makes the call of a number of tiles."""
    ks = cuda_lib.KeySchedule.from_triple(synth.key_triple(longest))
    x = torch.zeros(8192 * longest, dtype=torch.uint8, device="cuda")
    y = torch.empty_like(x)

    def call(tiles):
        a, b = x[:int(8192 * tiles)], y[:int(8192 * tiles)]
        if mode == "ecb":
            return lambda: cuda_lib.tdes_ecb_encrypt(ks, a, b)
        if mode == "ctr":
            return lambda: cuda_lib.tdes_ctr_crypt(ks, 5, 0, a, b)
        return lambda: cuda_lib.tdes_cbc_decrypt(ks, 9, a, b)

    return call


@pytest.mark.parametrize("mode", ["ecb", "ctr", "cbc_dec"])
@pytest.mark.parametrize("tail", [81, 120, 128])
def test_tails_in_a_row(cuda_lib, mode, tail):
    """Calls of one step of tiles (608) and a tail, one after another, take no
    longer than calls of 32 tiles more than the longest tail, all of them whole
    tiles."""
    step = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    call = _single_key(cuda_lib, mode, step + 160)
    r = _ratio(call(step + tail), call(step + 160), rows=50, rounds=20)
    assert r <= 1.08, r


@pytest.mark.parametrize("mode", ["ecb", "ctr", "cbc_dec"])
@pytest.mark.parametrize("before,more", [(300, 608), (700, 800)], ids=str)
def test_calls_after_uneven_ones(cuda_lib, mode, before, more):
    """A wide call that starts beside a call which loads the SMs unevenly: the two
    take no longer than with a larger, even call in its place."""
    call = _single_key(cuda_lib, mode, 1100)
    wide = call(1100)

    def pair(tiles):
        first = call(tiles)
        return lambda: (first(), wide())

    r = _ratio(pair(before), pair(more), rows=20, rounds=20)
    assert r <= 1.08, r


def test_small_calls_between_wide_ones(cuda_lib):
    """A call of 2048 blocks, 16 CTAs, that starts as a wide call's CTAs end: the two
    take little longer than with a call of one CTA (alone the larger takes 0.4 us
    longer)."""
    call = _single_key(cuda_lib, "ecb", 1100)
    wide, many, one = call(1100), call(2), call(1 / 16)
    r = _ratio(lambda: (many(), wide()), lambda: (one(), wide()), rows=20, rounds=20)
    assert r <= 1.15, r


@pytest.mark.parametrize("stages", [1, 3])
def test_ctr_on_8_byte_aligned_buffers(cuda_lib, stages):
    """CTR on buffers 8 bytes off a 16-byte boundary takes at most a third longer than
    on the boundary: 1.14 and 1.10 times, where loads wait for stores 1.98 and 1.47."""
    key, n = synth.key_triple(8), 8 * 2889442
    ks = cuda_lib.KeySchedule.des(key[:8]) if stages == 1 else cuda_lib.KeySchedule.from_triple(key)
    x = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")
    y = torch.empty_like(x)
    call = lambda off: lambda: cuda_lib.tdes_ctr_crypt(ks, 5, 7, x[off:off + n], y[off:off + n])  # noqa: E731
    r = _ratio(call(8), call(0), rounds=20)
    assert r <= 1.35, r


@pytest.mark.parametrize("nb,limit", [(3, 2.4), (50, 7.0), (200, 8.0)], ids=str)
def test_many_short_chains(cuda_lib, nb, limit):
    """20000 CBC encryptions of nb blocks against 32 of them: packed 32 to a warp
    they take 1.8, 5.5 and 6.7 times as long, where most go alone 3, 8.6 and 10.6."""
    n = 20000
    src = torch.zeros(8 * nb * n, dtype=torch.uint8, device="cuda")
    synth.fill_device(src, nb)
    dst = torch.empty_like(src)
    kt = cuda_lib.KeyTable(synth.key_triples(nb, 64))
    many, few = (cuda_lib.Batch(kt, [(4, i % 64, i << 32, src.data_ptr() + 8 * nb * i,
                                      dst.data_ptr() + 8 * nb * i, 8 * nb) for i in range(count)])
                 for count in (n, 32))
    r = _ratio(many.launch_graph, few.launch_graph, rounds=20)
    assert r <= limit, r


def test_single_des_chain(cuda_lib):
    """A single-DES CBC encryption takes little more than a third of an EDE3 one: 0.41
    of it, 0.44 where the permutations stand between the rounds of two blocks."""
    x = torch.zeros(8 * 2048, dtype=torch.uint8, device="cuda")
    key = synth.key_triple(6)
    des, ede = cuda_lib.KeySchedule.des(key[:8]), cuda_lib.KeySchedule.from_triple(key)
    y = torch.empty_like(x)
    r = _ratio(lambda: cuda_lib.tdes_cbc_encrypt(des, 3, x, y),
               lambda: cuda_lib.tdes_cbc_encrypt(ede, 3, x, y), rounds=20)
    assert r <= 0.425, r


# shares of the modes in tenths; the calls under many keys against under fewer: 1.08 and
# 1.21 times as long, where chains that want all warps run first 1.28 and 1.49
@pytest.mark.parametrize("msg,modes,many,few,limit", [
    (64, [4] * 10, 65536, 4096, 1.18), (256, [0, 0, 0, 0, 2, 2, 2, 3, 3, 4], 65536, 16384, 1.35)],
    ids=["chains", "mix"])
def test_uniform_chains_under_many_keys(cuda_lib, msg, modes, many, few, limit):
    n, T = 1 << 20, cuda_lib
    words = lambda stream: torch.from_numpy(synth.u64s(msg, n, stream).view(np.int64)).cuda()  # noqa: E731
    mode = torch.tensor(modes, dtype=torch.uint8, device="cuda")[(words(synth.STREAM_MODE) & 0xFFFF) * 10 >> 16]
    iv = words(synth.STREAM_IV) & -(1 << 32)
    src = torch.empty(n * msg, dtype=torch.uint8, device="cuda")
    synth.fill_device(src, msg)
    dst, pick, calls = torch.empty_like(src), words(synth.STREAM_KEYPICK), []
    for keys in (many, few):
        kt = T.KeyTable(synth.key_triples(msg, keys))
        index = (pick & (keys - 1)).to(torch.int32)
        need = T.tdes_uniform_scratch_bytes(kt, n, msg)
        buf = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
        scratch = buf[-buf.data_ptr() % 256:][:need]
        calls.append(lambda kt=kt, index=index, scratch=scratch: T.tdes_uniform_crypt(
            kt, index, mode, iv, src, dst, msg, scratch=scratch))
    r = _ratio(*calls, rounds=16)
    assert r <= limit, r
