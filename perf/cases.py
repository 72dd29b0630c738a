"""Performance cases of the verification library: what a verifier has it do, from one small
call to logs of 2^20 entries.

Every case is one call of a public entry point on a prepared batch:

  aver       poslo_aver with unit coefficients, POSLO-C or POSLO-F: one bit for the batch
  distill    poslo_distill, POSLO-F: the invalid entries and ccd^v
  distill_c  poslo_distill_c, POSLO-C: one bit per epoch, ccd^v, the umbrellas and ccd^i
  multi      poslo_aver_multi: many signers' logs in one batch
  stream     poslo_distill_stream: a log in page-locked host memory, chunk by chunk

A program keeps one context per instantiation for all its batches, as here.  Lengths, epoch
sizes, numbers of entries and shares of flipped entries are those of the benchmark and of the
tests (bench.py, tests/), or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_08781_gb300 import poslo

BPV_V, BPV_K = 64, 4   # BPV table and subset sizes of the benchmark's many-signer workload
TREE_SLACK = 1         # the seed tree has at least twice the epochs the batch spans


def listed():
    return [
        # a sensor's last few entries, checked as they arrive: launches and latency only
        _case("aver_f_60_host", op="aver", variant="F", n=60, lmin=32, lmax=256, host=True),
        # four epochs of a small log, as the benchmark's latency section has them
        _case("aver_c_1024_host", op="aver", variant="C", n=1024, lmin=64, lmax=64, host=True),
        _case("distill_f_1024_host", op="distill", variant="F", n=1024, lmin=64, lmax=64, flips=1, host=True),
        # an ordinary log of odd size whose last epoch is cut, a few entries flipped
        _case("distill_f_40k", op="distill", variant="F", n=40_013, lmin=32, lmax=256, flips=40),
        # the benchmark's step: a long log, all of it valid, and with 0.1 % of it flipped
        _case("distill_f_1m", op="distill", variant="F", n=1 << 20, lmin=32, lmax=256),
        _case("distill_f_1m_flips", op="distill", variant="F", n=1 << 20, lmin=32, lmax=256, flips=1049),
        # hashing alone: short entries of aggregate signatures, and long ones under AES
        _case("aver_c_1m_16b", op="aver", variant="C", n=1 << 20, lmin=16, lmax=16),
        _case("aver_c_1m_aes", op="aver", variant="C", n=1 << 20, lmin=32, lmax=256, aes=True),
        # cold storage of aggregate signatures distilled into umbrellas
        _case("distill_c_1m", op="distill_c", variant="C", n=1 << 20, lmin=32, lmax=256, flips=905, umbrellas=64),
        # a small batch of a service, from host memory, and a fleet's logs with a flipped few
        _case("multi_32_host", op="multi", variant="F", n=1_500, devices=32, lmin=32, lmax=256, flips=1, host=True),
        _case("multi_128", op="multi", variant="F", n=1_000_000, devices=128, lmin=32, lmax=256, flips=2),
        # a log larger than the chunk that fits the device's share, from page-locked memory
        _case("stream_1m_host", op="stream", variant="F", n=1_000_003, lmin=32, lmax=256, flips=1, chunk=1 << 18,
              host=True),
    ]


def _case(name=None, op="distill", variant="F", n=0, n2=256, lmin=32, lmax=256, flips=0, aes=False, host=False,
          umbrellas=0, devices=1, chunk=0):
    c = {"op": op, "variant": variant, "n": n, "n2": n2, "lmin": lmin, "lmax": lmax, "flips": flips, "aes": aes,
         "host": host, "umbrellas": umbrellas, "devices": devices, "chunk": chunk}
    if name is not None:
        c["name"] = name
    return c


def draw(rng):
    op = rng.choice(["aver", "aver", "distill", "distill", "distill", "distill_c", "multi", "stream"])
    lo = {"aver": 1, "distill": 1, "distill_c": 256, "multi": 64, "stream": 4096}[op]
    hi = 1_000_000 if op in ("multi", "stream") else 1 << 20
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))
    lmin, lmax = rng.choice([(8, 8), (16, 16), (32, 32), (64, 64), (1, 300), (32, 256), (32, 256)])
    variant = "C" if op == "distill_c" else rng.choice("CF") if op == "aver" else "F"
    n2 = rng.choice([256, 256, 64, 100])
    c = {"op": op, "variant": variant, "n2": n2, "lmin": lmin, "lmax": lmax, "aes": rng.random() < 0.25}
    if variant == "C":                              # whole epochs only
        n = min(max(n // n2, 1), (1 << 20) // n2) * n2
    if op in ("distill", "distill_c"):
        c["flips"] = rng.choice([0, 1, max(1, n // 1000)])
    if op == "distill_c":
        epochs = n // n2
        c["umbrellas"] = rng.choice([u for u in (1, 2, 4, 8, 16, 32, 64) if epochs % u == 0])
    if op == "multi":
        c["devices"] = max(2, min(256, n // rng.choice([8, 64, 2048])))
        c["flips"] = rng.choice([1, max(1, c["devices"] // 20)])
    if op == "stream":
        c["chunk"] = max(1024, n // rng.choice([2, 3, 5]))
        c["flips"] = rng.choice([1, max(1, n // 100_000)])
    c["host"] = op == "stream" or n * ((lmin + lmax) // 2 + 72) < (1 << 20) and rng.random() < 0.5
    return _case(n=n, **c)


# ------------------------------------------------------------------------------ inputs

_contexts: dict = {}


def _context(aes: bool) -> poslo.Context:
    """The program's verifier: one context per instantiation."""
    if aes not in _contexts:
        _contexts[aes] = poslo.Context(device=0, verifier_seed=bytes(range(7, 39)),
                                       instantiation=poslo.INST_AES if aes else poslo.INST_SHA256)
    return _contexts[aes]


def _messages(rng, case):
    n = case["n"]
    lens = rng.integers(case["lmin"], case["lmax"] + 1, n, dtype=np.int64)
    offs = np.zeros(n + 1, np.uint64)
    np.cumsum(lens, out=offs[1:])
    data = rng.integers(0, 256, max(int(offs[-1]), 1), dtype=np.uint8)
    return data, offs


def _flip_plan(case, seed, sizes=None):
    """(entry, position in [0, 1), mask) of the flipped entries.  AVer's outcome alternates with
    the seed; of many signers, or of POSLO-C epochs, `flips` have one flipped entry each."""
    rng = np.random.default_rng([seed, 2])
    if case["op"] == "multi":
        dev = np.sort(rng.choice(len(sizes), min(case["flips"], len(sizes)), replace=False))
        starts = np.concatenate([[0], np.cumsum(sizes)])
        idx = (starts[dev] + rng.random(len(dev)) * sizes[dev]).astype(np.int64)
    elif case["op"] == "distill_c":
        epochs = case["n"] // case["n2"]
        e = np.sort(rng.choice(epochs, min(case["flips"], epochs), replace=False))
        idx = e * case["n2"] + rng.integers(0, case["n2"], len(e))
    else:
        count = seed % 2 if case["op"] == "aver" else case["flips"]
        idx = np.sort(rng.choice(case["n"], min(count, case["n"]), replace=False)).astype(np.int64)
    return idx, rng.random(len(idx)), rng.integers(1, 256, len(idx), dtype=np.uint8)


def _flip(data, offs, plan):
    idx, pos, mask = plan
    out = data.copy()
    lens = (offs[idx + 1] - offs[idx]).astype(np.int64)
    out[offs[idx].astype(np.int64) + (pos * lens).astype(np.int64)] ^= mask
    return out


def _sizes(case, seed):
    """Entries per signer: log-uniform over three decades, scaled to the batch's n."""
    rng = np.random.default_rng([seed, 1])
    d = case["devices"]
    w = np.exp(rng.uniform(0, math.log(1000), d))
    sizes = np.maximum((w / w.sum() * (case["n"] - d)).astype(np.int64), 0) + 1
    sizes[int(np.argmax(sizes))] += case["n"] - int(sizes.sum())
    return sizes


def _scalars(rng, n):
    """n secret scalars below 2^252 (so below the group order), never zero."""
    b = rng.integers(0, 256, (n, 32), dtype=np.uint8)
    b[:, 31] &= 0x0F
    b[:, 0] |= 1
    return b


def _depth(epochs):
    return max(int(epochs - 1).bit_length(), 1) + TREE_SLACK


def _sign_f(ctx, rng, n2, first, msgs, offs):
    """A POSLO-F signer's key, disclosed seeds and signatures of entries first .. first + n - 1."""
    n = len(offs) - 1
    last = (first + n - 1) // n2
    D = _depth(last + 1)
    root = rng.bytes(16)
    y = _scalars(rng, 1)[0].tobytes()
    bpv_r = _scalars(rng, BPV_V)
    Y, bpv_R = ctx.keygen_f(y, bpv_r)
    subsets = rng.integers(0, BPV_V, (n, BPV_K), dtype=np.uint16)
    s, R = ctx.sign_f(y, root, D, n2, bpv_r, bpv_R, subsets, msgs, offs, first_index=first)
    return Y, ctx.disclose(root, D, last), s, R


def _sign_c(ctx, rng, n2, msgs, offs):
    epochs = (len(offs) - 1) // n2
    D = _depth(epochs)
    root, r = rng.bytes(16), rng.bytes(32)
    y = _scalars(rng, 1)[0].tobytes()
    Y, epoch_R = ctx.keygen_c(y, r, D, n2)
    s = ctx.sign_c(y, r, root, D, n2, msgs, offs, 0, epochs)
    return Y, ctx.disclose(root, D, epochs - 1), s, epoch_R[:32 * epochs].copy()


def _place(case, arrays):
    """The batch's arrays where the program holds them: device memory, or page-locked host
    memory for the streamed log and ordinary host memory for small calls."""
    if case["op"] == "stream":
        return [torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).pin_memory().numpy().view(a.dtype)
                for a in arrays]
    if case["host"]:
        return arrays
    return [torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).cuda() for a in arrays]


def prepare(case, seed):
    ctx = _context(case["aes"])
    rng = np.random.default_rng([seed, 0])
    data, offs = _messages(rng, case)
    n2 = case["n2"]
    state = {"ctx": ctx, "case": case}
    if case["op"] == "multi":
        sizes = _sizes(case, seed)
        starts = np.concatenate([[0], np.cumsum(sizes)])
        firsts = rng.integers(0, 4 * n2, len(sizes))
        keys, stacks, ss, Rs = [], [], [], []
        for d in range(len(sizes)):
            o = offs[starts[d]:starts[d + 1] + 1]
            part = data[int(o[0]):max(int(o[-1]), int(o[0]) + 1)]
            Y, ds, s, R = _sign_f(ctx, rng, n2, int(firsts[d]), part, o - o[0])
            keys.append(Y), stacks.append(ds), ss.append(s), Rs.append(R)
        data = _flip(data, offs, _flip_plan(case, seed, sizes))
        m, o, s, R = _place(case, [data, offs, np.concatenate(ss), np.concatenate(Rs)])
        state["args"] = (keys, sizes, firsts.astype(np.uint64), np.full(len(sizes), n2, np.uint32), stacks, m, o, s, R)
        return state
    if case["variant"] == "C":
        Y, ds, s, R = _sign_c(ctx, rng, n2, data, offs)
        if case["op"] == "aver":                    # the log's one signature
            s = np.frombuffer(ctx.agg(s, R)[0], np.uint8).copy()
        variant = poslo.VARIANT_C
    else:
        Y, ds, s, R = _sign_f(ctx, rng, n2, 0, data, offs)
        variant = poslo.VARIANT_F
    m, o, s, R = _place(case, [_flip(data, offs, _flip_plan(case, seed)), offs, s, R])
    state["batch"] = ctx.make_batch(variant, n2, Y, m, o, s, R, ds)
    return state


# ------------------------------------------------------------------------------ one pass

def _bytes(b):
    return np.frombuffer(b, np.uint8)


def run(state):
    ctx, case = state["ctx"], state["case"]
    op = case["op"]
    if op == "aver":
        return {"accept": ctx.aver(state["batch"])}
    if op == "distill":
        idx, s, R = ctx.distill(state["batch"])
        return {"invalid": idx, "ccd_s": _bytes(s), "ccd_R": _bytes(R)}
    if op == "distill_c":
        valid, ccd = ctx.distill_c(state["batch"], case["umbrellas"])
        return {"valid": np.array(valid), "invalid": np.array(ccd["invalid"], np.int64), "ccd_s": _bytes(ccd["s_v"]),
                "ccd_R": _bytes(ccd["R_v"]), "umbrellas": _bytes(b"".join(s + R for s, R in ccd["umbrellas"]))}
    if op == "multi":
        accept, pairs = ctx.aver_multi(*state["args"])
        return {"accept": accept, "pairs": pairs.reshape(-1)}
    accept, idx = ctx.distill_stream(state["batch"], case["chunk"])
    return {"accept": accept, "invalid": idx}


def work(case):
    """Inputs read once, outputs written once; the operations are 32-bit integer ones (the
    group arithmetic's multiply-adds and the hashing's logic), so none count as flops."""
    n, n2 = case["n"], case["n2"]
    b = n * ((case["lmin"] + case["lmax"]) / 2 + 8)                        # messages and offsets
    b += 64 * (n if case["variant"] == "F" else -(-n // n2))               # signatures
    if case["op"] in ("distill", "stream"):
        b += 8 * case["flips"] + 64
    if case["op"] == "distill_c":
        b += n // n2 + 64 * (case["umbrellas"] + 1) + 8 * case["flips"]
    if case["op"] == "multi":
        b += case["devices"] * (32 + 20 + 24 + 1) + 16 * case["flips"]
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """What follows from the flipped entries alone: the accept bits and the invalid lists (no
    floating-point numbers are computed anywhere).  The encoded sums have no such value here."""
    if case["op"] == "multi":
        sizes = _sizes(case, seed)
        idx = _flip_plan(case, seed, sizes)[0]
        rng = np.random.default_rng([seed, 0])
        _messages(rng, case)
        firsts = rng.integers(0, 4 * case["n2"], len(sizes))
        starts = np.concatenate([[0], np.cumsum(sizes)])
        dev = np.searchsorted(starts, idx, side="right") - 1
        accept = np.ones(len(sizes), bool)
        accept[dev] = False
        pairs = np.stack([dev, firsts[dev] + idx - starts[dev]], 1).reshape(-1).astype(np.uint64)
        return {"accept": accept, "pairs": pairs}
    idx = _flip_plan(case, seed)[0]
    if case["op"] == "aver":
        return {"accept": len(idx) == 0}
    if case["op"] == "distill":
        return {"invalid": idx.astype(np.uint64), "ccd_s": None, "ccd_R": None}
    if case["op"] == "stream":
        return {"accept": len(idx) == 0, "invalid": idx.astype(np.uint64)}
    bad = idx // case["n2"]
    valid = np.ones(case["n"] // case["n2"], bool)
    valid[bad] = False
    return {"valid": valid, "invalid": bad, "ccd_s": None, "ccd_R": None, "umbrellas": None}
