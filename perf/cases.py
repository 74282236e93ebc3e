"""Performance cases of the library: what its users have it do, from one
short seek to a 1 GiB decode, each through the public entry points of
``paper_2607_18541_gb300.aclz`` (and ``batched`` for many streams).

A case is a dict of plain values; ``prepare`` makes its inputs from the seed
alone, ``run`` makes one pass and returns the whole outputs, ``work`` counts
the bytes and operations the pass cannot do without, ``exact`` gives the
float outputs in 64 bits, ``draw`` gives more cases of the same ranges.

Kinds:

* ``sweep``   decode of the synthetic copy experiment (fixed match length)
* ``data``    decode of an encoded stream (FASTQ-like, word text, Markov bytes)
* ``batch``   many independent streams in one graph-captured decode
* ``seek``    one or more byte ranges of a resident, flattened text corpus
* ``upload``  container in host memory -> handle -> decoded bytes and their hash
* ``acle``    the same from an entropy-coded container, without the hash
* ``encode``  bytes in host memory -> container, parsed on the GPU
* ``mlp``     one training step of the threshold network (gradient and Adam)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_18541_gb300 import aclz, batched, synth

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30
PRESETS = {"base": aclz.ACLZ_PRESET_BASE, "tuned": aclz.ACLZ_PRESET_TUNED, "push": aclz.ACLZ_PRESET_PUSH}
# tokens per byte of the generated streams at 6/8/10/12, 12/16/24/32 and
# 16/24/32/48 and the share of bytes that are literals (means over seeds)
DENSITY = {("fastq", "base"): (0.058, 0.46), ("fastq", "tuned"): (0.0018, 0.97), ("fastq", "push"): (0.00013, 0.99),
           ("text", "base"): (0.065, 0.29), ("text", "tuned"): (0.005, 0.92), ("text", "push"): (0.0003, 0.99),
           ("markov", "base"): (0.0125, 0.72), ("markov", "tuned"): (0.0025, 0.90), ("markov", "push"): (0.0008, 0.96)}
IN, HID = 24, 64


def listed():
    return [
        # the paper's copy experiment at its largest: long matches, the
        # persistent schedule, as the benchmark runs it
        dict(name="sweep_1g_l1024", kind="sweep", total=GIB, L=1024, block=32 * KIB, G=32, ctas=2),
        # the same at short matches, library defaults
        dict(name="sweep_512m_l128", kind="sweep", total=512 * MIB, L=128, block=32 * KIB, G=32, ctas=0),
        # a sequencing file at 12/16/24/32: mostly literals, few waves
        dict(name="fastq_64m_tuned", kind="data", gen="fastq", n=64 * MIB, preset="tuned", block=16 * KIB,
             flatten=False, G=32),
        # text at the default 6/8/10/12: very short copies of copies,
        # decoded on the flattened schedule such chains need
        dict(name="text_32m_base_flat", kind="data", gen="text", n=32 * MIB, preset="base", block=64 * KIB,
             flatten=True, G=32),
        # a small record decoded by itself: latency and launches
        dict(name="markov_256k_base", kind="data", gen="markov", n=256 * KIB, preset="base", block=16 * KIB,
             flatten=False, G=32),
        # a request's worth of small streams decoded together
        dict(name="batch_64_streams", kind="batch", streams=64, lo=16 * KIB, hi=MIB, preset="tuned", block=16 * KIB,
             flatten=False, ctas=2),
        # the shortest call of a server: one page of the corpus
        dict(name="seek_16k", kind="seek", n=32 * MIB, requests=1, lo=16 * KIB, hi=16 * KIB),
        # one admitted batch of the serving loop
        dict(name="seek_batch_64", kind="seek", n=64 * MIB, requests=64, lo=16 * KIB, hi=4 * MIB),
        # receiving a container: upload, decode, verification hash
        dict(name="upload_verify_32m", kind="upload", gen="markov", n=32 * MIB, preset="tuned", block=32 * KIB,
             tagged=False),
        # receiving an entropy-coded container
        dict(name="upload_acle_64m", kind="acle", gen="fastq", n=64 * MIB, preset="tuned", block=16 * KIB),
        # producing a container
        dict(name="encode_text_16m", kind="encode", gen="text", n=16 * MIB, preset="tuned", block=64 * KIB, depth=64),
        # training the threshold network at its usual batch
        dict(name="mlp_step_256", kind="mlp", batch=256, K=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "data", "data", "data", "batch", "seek", "seek", "upload", "acle", "encode",
                       "mlp"])
    block = rng.choice([16, 32, 64]) * KIB
    if kind == "sweep":
        L = _log(rng, 32, 1024)
        most = 512 * MIB if L >= 128 else 128 * MIB
        return dict(kind=kind, total=_log(rng, 4 * MIB, most), L=L, block=block, G=rng.choice([32, 32, 32, 16]),
                    ctas=rng.choice([0, 2]))
    gen, preset = rng.choice(["fastq", "text", "markov"]), rng.choice(["base", "tuned", "tuned", "push"])
    if kind == "data":
        # streams whose copies copy copies are decoded flattened
        flatten = (preset == "base" and gen != "markov") or rng.random() < 0.3
        return dict(kind=kind, gen=gen, n=_log(rng, 16 * KIB, 48 * MIB), preset=preset, block=block,
                    flatten=flatten, G=rng.choice([32, 32, 32, 16]))
    if kind == "batch":
        return dict(kind=kind, streams=rng.randint(8, 96), lo=rng.randint(4, 32) * KIB, hi=rng.randint(100, 1024) * KIB,
                    preset="tuned", block=16 * KIB, flatten=rng.random() < 0.5, ctas=rng.choice([0, 2]))
    if kind == "seek":
        lo = _log(rng, 300, 256 * KIB)
        return dict(kind=kind, n=_log(rng, 4 * MIB, 64 * MIB), requests=_log(rng, 1, 128), lo=lo,
                    hi=_log(rng, lo, 1024 * KIB))
    if kind == "upload":
        tagged = rng.random() < 0.5
        if preset == "base" and gen != "markov":
            preset = "tuned"  # deep chains are uploaded flattened, not as waves
        return dict(kind=kind, gen=gen, n=_log(rng, MIB, 48 * MIB), preset=preset, block=block, tagged=tagged)
    if kind == "acle":
        return dict(kind=kind, gen=gen, n=_log(rng, MIB, 48 * MIB), preset="tuned", block=block)
    if kind == "encode":
        return dict(kind=kind, gen=gen, n=_log(rng, 64 * KIB, 16 * MIB), preset=preset, block=block,
                    depth=rng.choice([8, 64]))
    return dict(kind="mlp", batch=_log(rng, 32, 8192), K=rng.randint(2, 16))


# ---------------------------------------------------------------- inputs

def _bytes(gen, n, seed):
    if gen == "fastq":
        return synth.fastq(n, seed=seed)
    if gen == "text":
        return synth.wordtext(n, seed=seed, chunk_bytes=max(MIB, n // 8))
    return synth.markov2(n, seed=seed)


def _params(case, depth=64):
    p = aclz.aclz_encode_params_default(PRESETS[case["preset"]])
    p.block_size = case["block"]
    p.chain_depth = depth
    return p


def _container(case, seed):
    x = _bytes(case["gen"], case["n"], seed)
    return aclz.aclz_encode_gpu(x, _params(case))


def _room(n):
    return torch.zeros((n + 31) // 16 * 16, dtype=torch.uint8, device="cuda")


class _Handle:
    """An uploaded stream, freed with the state that holds it."""

    def __init__(self, container, flags=0):
        self.h = aclz.aclz_upload(container, flags=flags)

    def __del__(self):
        h, self.h = getattr(self, "h", None), None
        if h:
            aclz.aclz_free(h)


class _Batch:
    def __init__(self, containers, flatten, **cfg):
        self.dec = batched.BatchDecoder(containers, flatten=flatten)
        self.dec.out.zero_()
        self.dec.capture(**cfg)

    def __del__(self):
        dec, self.dec = getattr(self, "dec", None), None
        if dec is not None:
            torch.cuda.synchronize()
            dec.close()


def _mlp_state(case, seed):
    B, K = case["batch"], case["K"]
    P = IN * HID + HID + HID * HID + HID + HID * K + K
    r = np.random.RandomState(seed % (1 << 32))
    p = np.concatenate([r.randn(IN * HID) * math.sqrt(2 / IN), r.randn(HID) * 0.05,
                        r.randn(HID * HID) * math.sqrt(2 / HID), r.randn(HID) * 0.05,
                        r.randn(HID * K) * math.sqrt(1 / HID), r.randn(K) * 0.05]).astype(np.float32)
    m = (r.randn(P) * 1e-3).astype(np.float32)
    v = (r.rand(P) * 1e-5 + 1e-7).astype(np.float32)
    x = np.concatenate([r.rand(B, 16), r.randn(B, IN - 16)], axis=1).astype(np.float32)
    y = r.randint(0, K, B).astype(np.int32)
    return p, m, v, x, y


STEP, LR = 200, 1e-3
_SIZES = 2607  # the sizes of a batch's streams or requests are the case's own; their contents and places, the seed's


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "sweep":
        s = synth.copy_sweep(case["total"], case["block"], case["L"], seed=seed)
        c = aclz.aclz_pack(s.total, s.block_size, (4, 4, 4, 4), s.blk_ntok, s.lit_len, s.match_len, s.src, s.literals)
        st["handle"] = _Handle(c)
        st["out"], st["n"] = _room(case["total"]), case["total"]
        st["cfg"] = dict(G=case["G"], ctas_per_sm=case["ctas"])
    elif kind == "data":
        c = _container(case, seed)
        st["handle"] = _Handle(c, aclz.ACLZ_UPLOAD_FLATTEN if case["flatten"] else 0)
        st["out"], st["n"] = _room(case["n"]), case["n"]
        st["cfg"] = dict(G=case["G"])
    elif kind == "batch":
        sizes, _ = synth.stream_sizes(case["streams"], case["lo"], case["hi"], _SIZES)
        seeds = synth.rng_sequence(seed, case["streams"])
        model = synth.MarkovModel(seed)
        p = _params(case, depth=8)
        cs = [aclz.aclz_encode(synth.batch_stream(i, int(sizes[i]), int(seeds[i]), model), p)
              for i in range(case["streams"])]
        st["batch"] = _Batch(cs, case["flatten"], ctas_per_sm=case["ctas"])
    elif kind == "seek":
        c = _container(dict(gen="text", n=case["n"], preset="tuned", block=64 * KIB), seed)
        st["handle"] = _Handle(c, aclz.ACLZ_UPLOAD_FLATTEN)
        k = case["requests"]
        size = np.exp(np.random.RandomState(_SIZES).uniform(math.log(case["lo"]), math.log(case["hi"]), k))
        size = np.clip(size.astype(np.uint64), case["lo"], case["hi"])
        r = np.random.RandomState(seed % (1 << 32))
        lo = (r.rand(k) * (case["n"] - size)).astype(np.uint64)
        off = np.concatenate([[0], np.cumsum((size + 15) // 16 * 16)]).astype(np.uint64)
        st["out"] = _room(int(off[-1]))
        if k == 1:
            st["lo"], st["hi"] = int(lo[0]), int(lo[0] + size[0])
        else:
            table = torch.zeros(32 * k, dtype=torch.uint8).pin_memory()
            t = table.numpy().view(np.uint64).reshape(k, 4)
            t[:, 0], t[:, 1], t[:, 2] = lo, lo + size, off[:-1] + np.uint64(st["out"].data_ptr())
            st["table"] = table
    elif kind == "upload":
        c = _container(case, seed)
        if case["tagged"]:
            handle = _Handle(c)
            c = aclz.aclz_export(handle.h)
        st["container"] = torch.from_numpy(np.array(c)).pin_memory()
        st["out"], st["n"] = _room(case["n"]), case["n"]
    elif kind == "acle":
        st["container"] = aclz.aclz_acle_encode(_container(case, seed))
        st["out"], st["n"] = _room(case["n"]), case["n"]
    elif kind == "encode":
        st["x"], st["params"] = _bytes(case["gen"], case["n"], seed), _params(case, case["depth"])
        # the buffer a container is handed on in, as large as any container of this case
        tokens = case["n"] // 4 + 1 if case["preset"] == "base" else case["n"] // 16
        st["out"] = np.zeros(2 * case["n"] + 8 * tokens + 4096, dtype=np.uint8)
    else:
        p, m, v, x, y = (torch.from_numpy(a).cuda() for a in _mlp_state(case, seed))
        st.update(p=p, m=m, v=v, x=x, y=y, g=torch.empty_like(p), step=STEP,
                  loss=torch.empty(1, dtype=torch.float32, device="cuda"),
                  scratch=torch.empty(aclz.aclz_mlp_scratch_bytes(case["K"], case["batch"]), dtype=torch.uint8,
                                      device="cuda"))
    return st


# ------------------------------------------------------------------ pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("sweep", "data"):
        aclz.aclz_decode_all(st["handle"].h, st["out"], **st["cfg"])
        return st["out"][:st["n"]]
    if kind == "batch":
        dec = st["batch"].dec
        dec.replay()
        return dec.out[:dec.total]
    if kind == "seek":
        if case["requests"] == 1:
            aclz.aclz_decode_range(st["handle"].h, st["lo"], st["hi"], st["out"])
        else:
            aclz.aclz_decode_ranges_async(st["handle"].h, case["requests"], st["table"].data_ptr())
        return st["out"]
    if kind == "upload":
        h = aclz.aclz_upload(st["container"].numpy())
        try:
            aclz.aclz_decode_all(h, st["out"])
            f = aclz.aclz_fnv(st["out"], st["n"])
        finally:
            aclz.aclz_free(h)
        return st["out"][:st["n"]], f >> 32, f & 0xffffffff
    if kind == "acle":
        h = aclz.aclz_upload_acle(st["container"])
        try:
            aclz.aclz_decode_all(h, st["out"])
            if aclz.aclz_device_status(h) != aclz.ACLZ_OK:
                raise RuntimeError("decode reported a device error")
        finally:
            aclz.aclz_free(h)
        return st["out"][:st["n"]]
    if kind == "encode":
        c = aclz.aclz_encode_gpu(st["x"], st["params"])
        st["out"][:c.size] = c
        return st["out"], c.size
    K = case["K"]
    aclz.aclz_mlp_grad(st["p"], K, st["x"], st["y"], case["batch"], st["g"], st["loss"], st["scratch"])
    aclz.aclz_mlp_adam(st["p"], st["m"], st["v"], st["g"], K, st["step"], LR)
    st["step"] += 1
    return dict(g=st["g"], loss=st["loss"], m=st["m"], p=st["p"], v=st["v"])


# ------------------------------------------------------------------ work

def _decode_bytes(n, tokens, literals):
    # 16 B per token, literals and match sources read, output written
    return 16 * tokens + literals + (n - literals) + n


def _container_bytes(n, tokens, literals, block):
    return 64 + 32 * ((n + block - 1) // block) + 16 * tokens + literals


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        tokens = case["total"] / (case["L"] + 4)
        return {"bytes": _decode_bytes(case["total"], tokens, 4 * tokens), "flops": 0}
    if kind == "mlp":
        B, K = case["batch"], case["K"]
        P = IN * HID + HID + HID * HID + HID + HID * K + K
        # parameters and moments read and written, gradient written, batch read
        return {"bytes": 4 * (7 * P + B * (IN + 1) + 1), "flops": 6 * B * (IN * HID + HID * HID + HID * K) + 12 * P}
    if kind == "seek":
        mean = case["lo"] if case["hi"] == case["lo"] else (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        d, f = DENSITY[("text", "tuned")]
        return {"bytes": case["requests"] * mean * (2 + 16 * d), "flops": 0}
    if kind == "batch":
        n = case["streams"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": _decode_bytes(n, 0.002 * n, 0.93 * n), "flops": 0}
    n = case["n"]
    d, f = DENSITY[(case["gen"], case["preset"])]
    tokens, literals = d * n, f * n
    size = _container_bytes(n, tokens, literals, case["block"])
    if kind == "data":
        return {"bytes": _decode_bytes(n, tokens, literals), "flops": 0}
    if kind == "upload":
        # container across the link and into memory, decode, hash
        return {"bytes": 2 * size + _decode_bytes(n, tokens, literals) + n, "flops": 0}
    if kind == "acle":
        # coded container in, v1 arrays written, decode
        return {"bytes": 0.5 * n + size + _decode_bytes(n, tokens, literals), "flops": 0}
    return {"bytes": n + size, "flops": 0}  # encode


# ----------------------------------------------------------------- exact

def exact(case, seed):
    """The float outputs in 64 bits (the other kinds return bytes)."""
    if case["kind"] != "mlp":
        return None
    p, m, v, x, y = (a.astype(np.float64) if a.dtype != np.int32 else a for a in _mlp_state(case, seed))
    B, K = case["batch"], case["K"]
    shapes = [(IN, HID), (HID,), (HID, HID), (HID,), (HID, K), (K,)]
    W, at = [], 0
    for s in shapes:
        n = int(np.prod(s))
        W.append(p[at:at + n].reshape(s))
        at += n
    W1, b1, W2, b2, W3, b3 = W
    h1 = np.maximum(x @ W1 + b1, 0)
    h2 = np.maximum(h1 @ W2 + b2, 0)
    z = h2 @ W3 + b3
    z = z - z.max(axis=1, keepdims=True)
    s = np.exp(z)
    q = s / s.sum(axis=1, keepdims=True)
    loss = float(np.mean(np.log(s.sum(axis=1)) - z[np.arange(B), y]))
    dz = q.copy()
    dz[np.arange(B), y] -= 1
    dz /= B
    d2 = (dz @ W3.T) * (h2 > 0)
    d1 = (d2 @ W2.T) * (h1 > 0)
    g = np.concatenate([a.reshape(-1) for a in (x.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ dz, dz.sum(0))])
    m = 0.9 * m + 0.1 * g
    v = 0.999 * v + 0.001 * g * g
    p = p - LR * (m / (1 - 0.9 ** STEP)) / (np.sqrt(v / (1 - 0.999 ** STEP)) + 1e-8)
    return dict(g=g, loss=np.array([loss]), m=m, p=p, v=v)
