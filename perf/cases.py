"""Performance cases of the 3DES framework: what its users call, at the sizes they call it with.

Every case goes through the public Python entry points of
``paper_2007_10752_gb300.tdes`` with the handles a program keeps (key
schedules, key tables, batch plans, contexts, servers) made beforehand.
Payloads, keys, IVs, lengths and modes are drawn from the seed with the
package's own SplitMix64 generator: uniform random bytes, random key triples,
log-uniform lengths and the mode mixes of the repository's workloads.
"""
import math

import numpy as np
import torch

from paper_2007_10752_gb300 import synth, tdes

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30

# mode mixes of the repository's workloads, as (mode, share)
MIX_ALL = ((0, 0.4), (2, 0.3), (3, 0.2), (4, 0.1))  # ECB, CTR, CBC-decrypt, CBC-encrypt
MIX_PARALLEL = ((0, 4 / 9), (2, 3 / 9), (3, 2 / 9))  # without the serial CBC encryption
MIX_SERVE = ((0, 1 / 3), (2, 1 / 3), (3, 1 / 3))


def listed():
    return [
        # The smallest file of the paper's table (4 blocks): one call's latency.
        dict(name="ecb_32b", kind="ecb", nbytes=32),
        # The paper's largest file and the plain single-launch workload: 1 MiB, there and back.
        dict(name="ecb_1mib", kind="ecb", nbytes=1 * MIB, both=True),
        # An ordinary file or record batch, not a multiple of any tile, decrypted.
        dict(name="ecb_dec_9mb", kind="ecb", nbytes=9000008, decrypt=True),
        # The headline workload: one 1 GiB buffer under one triple.
        dict(name="ecb_1gib", kind="ecb", nbytes=1 * GIB),
        # A CTR stream segment starting at an odd counter, ragged end.
        dict(name="ctr_40mb", kind="ctr", nbytes=40000072, ctr0=1000001),
        # Decrypting a large CBC file into another buffer.
        dict(name="cbc_dec_200mb", kind="cbc_dec", nbytes=200000024),
        # Encrypting one CBC record: a serial chain of 2048 blocks.
        dict(name="cbc_enc_16kib", kind="cbc_enc", nbytes=16 * KIB),
        # Messages of 64 B to 4 MiB, each under its own triple, in the modes
        # that are parallel inside a message; a plan replayed as a CUDA graph.
        dict(name="batch_4096", kind="batch", count=4096, lo=64, hi=4 * MIB, parallel=True),
        # Small records in all four modes handed to a batch context for a ticket and waited for.
        dict(name="ctx_4096_small", kind="ctx", count=4096, lo=64, hi=4 * KIB),
        # 64-byte messages under many triples, planned on the device.
        dict(name="uniform_64m_64b", kind="uniform", count=1 << 26, msg=64, keys=16384),
        # A burst of requests through the continuous-batching server: 80% small, 20% large.
        dict(name="serve_1024", kind="serve", count=1024, keys=16384),
        # Data that lives on the host: 256 MiB of pinned memory, in place.
        dict(name="host_256mib", kind="host", nbytes=256 * MIB),
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["ecb", "ecb", "ctr", "ctr", "cbc_dec", "cbc_dec", "cbc_enc", "batch", "ctx",
                       "uniform", "serve", "host"])
    if kind in ("ecb", "ctr", "cbc_dec"):
        c = dict(kind=kind, nbytes=8 * _log(rng, 4, GIB // 8))
        c["single_des"] = rng.random() < 0.15
        c["offset8"] = rng.random() < 0.15  # a buffer that is only 8-byte aligned
        c["in_place"] = rng.random() < 0.3
        if kind == "ecb":
            c["decrypt"] = rng.random() < 0.5
        if kind == "ctr":
            c["ctr0"] = rng.choice([0, 1, rng.randrange(1 << 20)])
        return c
    if kind == "cbc_enc":
        return dict(kind=kind, nbytes=8 * _log(rng, 1, 8 * KIB), single_des=rng.random() < 0.15)
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 64, 4096), lo=64, hi=_log(rng, 4 * KIB, 4 * MIB),
                    parallel=True)
    if kind == "ctx":
        return dict(kind=kind, count=_log(rng, 256, 16384), lo=64, hi=_log(rng, 256, 8 * KIB))
    if kind == "uniform":
        msg = rng.choice([8, 16, 64, 64, 128, 200, 256])
        return dict(kind=kind, count=_log(rng, 1 << 14, min(1 << 26, (1 << 32) // msg) - 1) | 1, msg=msg,
                    keys=1 << rng.randrange(4, 17))
    if kind == "serve":
        return dict(kind=kind, count=_log(rng, 64, 1024), keys=16384)
    return dict(kind=kind, nbytes=8 * _log(rng, MIB // 8, 256 * MIB // 8))


def _payload(nbytes, seed):
    x = torch.empty((nbytes + 7) // 8 * 8, dtype=torch.uint8, device="cuda")
    synth.fill_device(x, seed)
    return x


def _modes(seed, n, mix):
    m = np.array([m for m, _ in mix], dtype=np.uint32)
    return m[synth.categorical(seed, n, [p for _, p in mix], synth.STREAM_MODE)]


def _serve_lengths(seed, n):
    """80% uniform in 64 B..4 KiB, 20% log-uniform in 64 KiB..16 MiB."""
    small = synth.categorical(seed, n, [0.8, 0.2], synth.STREAM_SIZECLASS) == 0
    u = synth.uniform01(seed, n, synth.STREAM_LENGTH)
    lens = np.where(small, 64 + u * (4 * KIB - 64), 64 * KIB * np.exp(u * math.log(256.0)))
    return lens.astype(np.int64) // 8 * 8


def _messages(case):
    """(lengths, modes) of a batch, a context's batch or a server's burst; the
    same for every seed, so that a case is the same work each time."""
    n = case["count"]
    if case["kind"] == "serve":
        return _serve_lengths(11, n), _modes(11, n, MIX_SERVE)
    mix = MIX_PARALLEL if case.get("parallel") else MIX_ALL
    return synth.log_uniform_lengths(11, n, case["lo"], case["hi"]), _modes(11, n, mix)


def _batch(case, seed, n_keys):
    lens, modes = _messages(case)
    n = len(lens)
    offs = np.concatenate([[0], np.cumsum((lens + 15) // 16 * 16)]).astype(np.uint64)
    src = _payload(int(offs[-1]), seed)
    dst = torch.zeros_like(src)
    ivs = synth.u64s(seed, n, synth.STREAM_IV)
    d = np.zeros(n, dtype=tdes.DESC_DTYPE)
    d["mode"] = modes
    d["key_index"] = (synth.u64s(seed, n, synth.STREAM_KEYPICK) % np.uint64(n_keys)).astype(np.uint32)
    d["iv_or_ctr"] = np.where(modes == 2, ivs & np.uint64(0xFFFFFFFF00000000), ivs)
    d["in_ptr"] = np.uint64(src.data_ptr()) + offs[:-1]
    d["out_ptr"] = np.uint64(dst.data_ptr()) + offs[:-1]
    d["nbytes"] = lens.astype(np.uint64)
    return src, dst, tdes.KeyTable(synth.key_triples(seed, n_keys)), d


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("ecb", "ctr", "cbc_dec", "cbc_enc", "host"):
        triple = synth.key_triple(seed)
        s["ks"] = (tdes.KeySchedule.des(triple[:8]) if case.get("single_des")
                   else tdes.KeySchedule.from_triple(triple))
        s["iv"] = synth.iv64(seed)
        n = case["nbytes"]
    if kind == "host":
        s["host"] = torch.empty(n, dtype=torch.uint8, pin_memory=True)
        s["host"].copy_(_payload(n, seed)[:n])
        s["dev"] = torch.empty(512 * MIB, dtype=torch.uint8, device="cuda")
    elif kind in ("ecb", "ctr", "cbc_dec", "cbc_enc"):
        o = 8 if case.get("offset8") else 0
        s["x"] = _payload(n + o, seed)[o:]
        s["y"] = s["x"] if case.get("in_place") else torch.zeros(n + o, dtype=torch.uint8,
                                                                 device="cuda")[o:]
        if case.get("both"):
            s["z"] = torch.zeros_like(s["x"])
    elif kind == "batch":
        s["src"], s["dst"], s["kt"], d = _batch(case, seed, case["count"])
        s["plan"] = tdes.Batch(s["kt"], d)
    elif kind == "ctx":
        s["src"], s["dst"], s["kt"], s["descs"] = _batch(case, seed, case["count"])
        s["ctx"] = tdes.Ctx(s["kt"])
    elif kind == "serve":
        s["src"], s["dst"], s["kt"], d = _batch(case, seed, case["keys"])
        s["entries"] = [tuple(int(v) for v in row) for row in d.tolist()]
        s["server"] = tdes.Server(s["kt"])
    else:
        n, m = case["count"], case["msg"]
        keys = case["keys"]

        def words(stream):
            w = torch.empty(n, dtype=torch.int64, device="cuda")
            synth.fill_device(w.view(torch.uint8), seed, stream)
            return w

        s["kt"] = tdes.KeyTable(synth.key_triples(seed, keys))
        s["key_index"] = (words(synth.STREAM_KEYPICK) & (keys - 1)).to(torch.int32)
        pick = (words(synth.STREAM_MODE) & 0xFFFF) * 10 >> 16  # 0..9, evenly
        s["mode"] = torch.tensor([0, 0, 0, 0, 2, 2, 2, 3, 3, 4], dtype=torch.uint8,
                                 device="cuda")[pick]
        iv = words(synth.STREAM_IV)
        s["iv"] = torch.where(s["mode"] == 2, iv & -(1 << 32), iv)
        s["src"] = _payload(n * m, seed)
        s["dst"] = torch.zeros_like(s["src"])
        need = tdes.tdes_uniform_scratch_bytes(s["kt"], n, m)
        buf = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
        off = -buf.data_ptr() % 256
        s["scratch"] = buf[off:off + need]
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "ecb":
        call = tdes.tdes_ecb_decrypt if case.get("decrypt") else tdes.tdes_ecb_encrypt
        y = call(s["ks"], s["x"], s["y"])
        return [y, tdes.tdes_ecb_decrypt(s["ks"], y, s["z"])] if case.get("both") else y
    if kind == "ctr":
        return tdes.tdes_ctr_crypt(s["ks"], s["iv"] >> 32, case["ctr0"], s["x"], s["y"])
    if kind == "cbc_dec":
        return tdes.tdes_cbc_decrypt(s["ks"], s["iv"], s["x"], s["y"])
    if kind == "cbc_enc":
        return tdes.tdes_cbc_encrypt(s["ks"], s["iv"], s["x"], s["y"])
    if kind == "host":
        return tdes.tdes_ecb_crypt_host(s["ks"], False, s["host"], s["host"], s["dev"])
    if kind == "batch":
        s["plan"].launch_graph()
        return s["dst"]
    if kind == "ctx":
        ticket = s["ctx"].submit(s["descs"])
        status = s["ctx"].wait(ticket)
        s["ctx"].release(ticket)
        return [s["dst"], status]
    if kind == "serve":
        group = s["server"].submit_group(s["entries"])
        return [s["dst"], s["server"].wait_group(group)]
    tdes.tdes_uniform_crypt(s["kt"], s["key_index"], s["mode"], s["iv"], s["src"], s["dst"],
                            case["msg"], scratch=s["scratch"])
    return s["dst"]


def work(case):
    """Payload in and payload out; per-message key index, mode and IV where the call takes them."""
    kind = case["kind"]
    if kind in ("batch", "ctx", "serve"):
        lens, _ = _messages(case)
        return {"bytes": 2 * int(lens.sum()) + 40 * len(lens), "flops": 0}
    if kind == "uniform":
        return {"bytes": case["count"] * (2 * case["msg"] + 13), "flops": 0}
    return {"bytes": (4 if case.get("both") else 2) * case["nbytes"], "flops": 0}
