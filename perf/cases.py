"""What users have this library do, as timed cases (through the Python binding).

Each case is one call a user's program makes, with the state such a program
keeps (keys, device buffers, workspace, a reusable batch) built beforehand by
prepare().  Sizes are those of params.py, the benchmark and the tests: the
n = 630 / N = 1024 key set with 1 to 4 rows, the same inputs in the
single-polynomial layout (N = 4096), the n = 750 / N = 2048 key set with up to
8 rows, the uneven mix over both, the two-round evaluation of arbitrary
functions at the plaintext-size sweep's key sets (N = 2048 and 16384), the key
switch alone, and the toy key set.  All outputs are whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_12441_gb300 import api, params as P, synth

# the sweep's single-polynomial layout at log t = 8 (two-pass ring degrees)
KEYS_SWEEP_N16384 = P.KeyParams(n=512, N=16384, Q=P.KEYS_SWEEP_N2048.Q, log2_B=15, l_B=4,
                                log2_Bks=5, l_ks=8)

KEYS = {"toy": P.KEYS_TOY, "n1024": P.KEYS_N1024, "n2048": P.KEYS_N2048, "n4096": P.KEYS_N4096,
        "sweep2048": P.KEYS_SWEEP_N2048, "sweep16384": KEYS_SWEEP_N16384}

# (m, log2 t) of the uneven mix, with the key set of each
MIX = [("n1024", 1, 8), ("n1024", 2, 9), ("n1024", 4, 10), ("n2048", 2, 11), ("n2048", 4, 12), ("n2048", 8, 13)]


def listed() -> list[dict]:
    return [
        # the toy parameter set, all of its 32 messages in one call: the smallest bootstrap
        {"name": "toy_32", "kind": "boot", "keys": "toy", "m": 2, "logt": 5, "count": 32},
        # one ciphertext per call (the plain form of the benchmark): pure latency
        {"name": "plain_one", "kind": "boot", "keys": "n1024", "m": 4, "logt": 10, "count": 1},
        # the headline batch at a quarter of its size, a ragged last wave
        {"name": "batch_m4", "kind": "boot", "keys": "n1024", "m": 4, "logt": 10, "count": 1000},
        # the smallest plaintext of the mix: one row per ciphertext
        {"name": "batch_m1", "kind": "boot", "keys": "n1024", "m": 1, "logt": 8, "count": 1200},
        # the single-polynomial layout (m = 1, N = 4096) the headline batch is compared with
        {"name": "single_poly", "kind": "boot", "keys": "n4096", "m": 1, "logt": 10, "count": 300},
        # large plaintexts, random and identity tables, more jobs than SMs
        {"name": "large_m8", "kind": "boot", "keys": "n2048", "m": 8, "logt": 13, "count": 200},
        # a small served batch of the large-plaintext set: host buffers, copies inside the call
        {"name": "served_8", "kind": "host", "keys": "n2048", "m": 8, "logt": 13, "count": 8},
        # the uneven mix over two resident key sets: persistent kernels replayed from a CUDA graph
        {"name": "uneven", "kind": "mix", "count": 900},
        # an arbitrary function by two rounds, the sweep's BootMMPM row at log t = 7
        {"name": "two_round", "kind": "two_round", "keys": "sweep2048", "m": 4, "logt": 7, "count": 150},
        # the sweep's single-polynomial row at log t = 8 (ring degree 16384)
        {"name": "two_round_big", "kind": "two_round", "keys": "sweep16384", "m": 1, "logt": 8, "count": 40},
        # key switching alone, a batch of samples
        {"name": "key_switch", "kind": "ks", "keys": "n1024", "count": 2000},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["boot", "boot", "boot", "host", "mix", "two_round", "two_round_big", "ks"])
    if kind in ("boot", "host"):
        keys = rng.choice(["n1024", "n1024", "n2048", "n2048", "n4096", "toy"])
        m = {"n1024": rng.randint(1, 6), "n2048": rng.randint(1, 9), "n4096": 1, "toy": rng.randint(1, 4)}[keys]
        logt = rng.randint(4, {"n1024": 8, "n2048": 10, "n4096": 10, "toy": 4}[keys] + m.bit_length() - 1)
        top = {"n1024": 4200, "n2048": 1400, "n4096": 900, "toy": 2000}[keys] // m
        return {"kind": kind, "keys": keys, "m": m, "logt": logt, "count": _log_int(rng, 1, top)}
    if kind == "mix":
        return {"kind": "mix", "count": _log_int(rng, 6, 1200)}
    if kind == "two_round":
        m = 1 << rng.randint(0, 4)
        return {"kind": "two_round", "keys": "sweep2048", "m": m, "logt": rng.randint(3, 4 + m.bit_length()),
                "count": _log_int(rng, 1, 800 // m)}
    if kind == "two_round_big":
        return {"kind": "two_round", "keys": "sweep16384", "m": 1, "logt": rng.randint(5, 8),
                "count": _log_int(rng, 1, 60)}
    return {"kind": "ks", "keys": rng.choice(["n1024", "n2048", "n4096"]), "count": _log_int(rng, 1, 4000)}


def _luts(t: int, count: int, rng: np.random.Generator, mixed: bool) -> tuple[np.ndarray, np.ndarray]:
    lo = rng.integers(0, t, (count, t // 2), dtype=np.int64)
    ident = np.zeros(count, bool)
    if mixed:
        ident[1::2] = True
        lo[1::2] = np.arange(t // 2)
    return np.concatenate([lo, (t - lo) % t], axis=1).astype(np.uint32), ident


def _jobs(sk, kp, ki, m, t, count, rng, mixed, in0=0, lut0=0):
    """Job records, ciphertexts and tables of one (key set, shape) group."""
    luts, ident = _luts(t, count, rng, mixed)
    msg = rng.integers(0, t, count).astype(np.uint32)
    msg[ident] %= t // 2
    ct = api.bm_encrypt_seeded(sk, 2 * kp.N * m, t, msg, int(rng.integers(1 << 62)))
    W = kp.n + 1
    off = in0 + np.arange(count) * W
    return api.make_jobs(ki, m, t, off, lut0 + np.arange(count) * t, off), ct.ravel(), luts.ravel()


def prepare(case: dict, seed: int) -> dict:
    rng = np.random.default_rng([seed, 12441])
    key_seed = int(rng.integers(1 << 62))
    kind, count = case["kind"], case["count"]
    if kind == "mix":
        names = ["n1024", "n2048"]
    else:
        names = [case["keys"]]
    sets = [(KEYS[k],) + api.bm_keygen_seeded(KEYS[k], key_seed) for k in names]
    keys = [ek for _, _, ek in sets]
    kp, sk, ek = sets[0]
    st = {"kind": kind, "keys": keys, "count": count}
    if kind == "ks":
        lwe = rng.integers(0, kp.Q, count * (kp.N + 1), dtype=np.uint64)
        st["in"] = api.to_device_u64(lwe)
        st["out"] = torch.zeros(count * (kp.n + 1), dtype=torch.int64, device="cuda")
        return st
    if kind == "two_round":
        m, t = case["m"], 1 << case["logt"]
        q = 2 * kp.N * m
        x = rng.integers(0, 2 * t, count).astype(np.uint32)
        ct = api.bm_encrypt_seeded(sk, q, 2 * t, x, int(rng.integers(1 << 62)))
        st.update(m=m, t=t, q=q, f=api.to_device_u32(rng.integers(0, t, count * t).astype(np.uint32)))
        st["in"] = api.to_device_u64(ct.ravel())
        st["out"] = torch.zeros(count * (kp.n + 1), dtype=torch.int64, device="cuda")
        st["ws"] = api.workspace(api.bm_arbitrary_workspace_bytes(ek, m, t, count))
        return st
    if kind == "mix":
        # Zipf(1.2) shares of the six shapes, every shape at least once, jobs interleaved
        w = np.arange(1, len(MIX) + 1) ** -1.2
        counts = np.maximum(np.floor(count * w / w.sum()).astype(int), 1)
        parts, in0, lut0 = [], 0, 0
        for (kn, m, logt), c in zip(MIX, counts):
            ki = names.index(kn)
            part = _jobs(sets[ki][1], sets[ki][0], ki, m, 1 << logt, int(c), rng, False, in0, lut0)
            parts.append(part)
            in0 += part[1].size
            lut0 += part[2].size
        jobs = np.concatenate([p[0] for p in parts])
        jobs = jobs[rng.permutation(len(jobs))]
        ct, luts = np.concatenate([p[1] for p in parts]), np.concatenate([p[2] for p in parts])
    else:
        jobs, ct, luts = _jobs(sk, kp, 0, case["m"], 1 << case["logt"], count, rng, case["keys"] == "n2048")
    st["jobs"] = jobs
    if kind == "host":
        st["in"] = torch.from_numpy(ct.view(np.int64)).pin_memory()
        st["lut"] = torch.from_numpy(luts.view(np.int32)).pin_memory()
        st["out"] = torch.zeros(ct.size, dtype=torch.int64).pin_memory()
        st["ws"] = api.workspace(api.bm_workspace_bytes(keys, jobs) + api.bm_host_staging_bytes(keys, jobs))
        return st
    st["in"], st["lut"] = api.to_device_u64(ct), api.to_device_u32(luts)
    st["out"] = torch.zeros(ct.size, dtype=torch.int64, device="cuda")
    st["ws"] = api.workspace(api.bm_workspace_bytes(keys, jobs))
    if kind == "mix":
        # the executor a server keeps: job table uploaded once, launches replayed from a graph
        st["stream"] = torch.cuda.Stream()
        st["batch"] = api.Batch(keys, jobs, st["in"], st["lut"], st["out"], st["ws"],
                                api.BATCH_GRAPH | api.BATCH_PERSISTENT)
        torch.cuda.synchronize()
    return st


def run(st: dict):
    kind = st["kind"]
    if kind == "boot":
        api.bm_bootstrap_batch(st["keys"], st["jobs"], st["in"], st["lut"], st["out"], st["ws"])
    elif kind == "host":
        api.bm_bootstrap_batch_host(st["keys"], st["jobs"], st["in"], st["lut"], st["out"], st["ws"])
    elif kind == "mix":
        # the batch runs on its own stream, ordered with the caller's
        s = st["stream"]
        s.wait_stream(torch.cuda.current_stream())
        st["batch"].run(s)
        torch.cuda.current_stream().wait_stream(s)
    elif kind == "two_round":
        api.bm_bootstrap_arbitrary(st["keys"][0], st["m"], st["t"], st["q"], st["f"], st["count"], st["in"],
                                   st["out"], st["ws"])
    else:
        api.bm_key_switch(st["keys"][0], st["in"], st["count"], st["out"])
    return st["out"]


def _boot_work(kp, m: int, t: int, count: int) -> tuple[float, float]:
    """64-bit modular products (transforms of the 4 l_B digit polynomials and
    the two sums per row, products with the key rows) and bytes in and out."""
    lg = kp.N.bit_length() - 1
    mul = kp.n * m * ((4 * kp.l_B + 2) * (kp.N // 2) * lg + 8 * kp.l_B * kp.N)
    return count * mul, count * (16 * (kp.n + 1) + 4 * t)


def _key_bytes(kp) -> tuple[int, int]:
    bsk = kp.n * 2 * 2 * kp.l_B * 2 * kp.N * 8
    ksk = kp.N * kp.l_ks * (kp.Bks - 1) * (kp.n + 1) * 8
    return bsk, ksk


def _ks_bytes(kp, count: int) -> int:
    # the key rows the digits select (a zero digit selects none), at most the whole key
    sel = kp.N * kp.l_ks * (kp.Bks - 1) / kp.Bks * (kp.n + 1) * 8
    return int(min(count * sel, _key_bytes(kp)[1]))


def work(case: dict) -> dict:
    kind, count = case["kind"], case["count"]
    if kind == "mix":
        w = np.arange(1, len(MIX) + 1) ** -1.2
        counts = np.maximum(np.floor(count * w / w.sum()).astype(int), 1)
        flops = nbytes = 0
        for kn in ("n1024", "n2048"):
            c = sum(int(x) for (k, _, _), x in zip(MIX, counts) if k == kn)
            nbytes += _key_bytes(KEYS[kn])[0] + _ks_bytes(KEYS[kn], c)
        for (kn, m, logt), c in zip(MIX, counts):
            f, b = _boot_work(KEYS[kn], m, 1 << logt, int(c))
            flops, nbytes = flops + f, nbytes + b
        return {"bytes": nbytes, "flops": flops}
    kp = KEYS[case["keys"]]
    if kind == "ks":
        return {"bytes": _ks_bytes(kp, count) + count * 8 * (kp.N + kp.n + 2),
                "flops": count * kp.N * kp.l_ks * (kp.n + 1)}
    rounds = 2 if kind == "two_round" else 1
    f, b = _boot_work(kp, case["m"], 1 << case["logt"], count)
    return {"bytes": _key_bytes(kp)[0] + _ks_bytes(kp, count) + b, "flops": rounds * f}


def exact(case: dict, seed: int):
    # Every output is a whole number: the bits of a ciphertext under keys that
    # stay inside the library.
    return None
