"""Measured cases: what a user of the library has it do, through its public entry points.

A case is one of these kinds of work, with its sizes:

  round     one whole aggregation round on device data: every client packs and encrypts its update, the
            server forms the weighted sum of the ciphertexts (and the average of the plaintext remainder
            when a mask is used), the result is decrypted and merged into one model
  host      the same round from host buffers through the one-call entry point (copies included)
  encrypt   one client's half: pack an update and encrypt it
  server    the server's half: weighted sum of all clients' ciphertexts with the rescale
  open      the receiving half: decrypt the aggregate and unpack it
  mask      selection of the largest sensitivity scores and its index list
  ntt       the standalone batched transforms, forward and inverse

Ring degrees and primes are the parameter sets that the repository's workloads, tests and kernel sweep
use: 60/40/60 bits on N = 8192, 60/40/40/60 on N = 16384, 60/45x4/60 on N = 32768, and twelve 60-bit or
45-bit primes for the kernel sweep up to N = 65536.
"""
from __future__ import annotations

import math

import torch

import paper_2303_10837_b200 as he

# largest primes below 2^b with q = 1 (mod 2N), descending, distinct
SETS = {
    "60-40-60": (0xfffffffffffc001, 0xfffffdc001, 0xffffffffffe8001),
    "60-40-40-60": (0xffffffffffe8001, 0xffffe80001, 0xffffca8001, 0xffffffffffd8001),
    "60-45x4-60": (0xffffffffffc0001, 0x1fffffcf0001, 0x1fffffc20001, 0x1fffffbf0001, 0x1fffffb10001,
                   0xfffffffff840001),
    # = 1 (mod 2^17): good for every ring; a case takes the first `limbs` of them
    "60": (0xffffffffffc0001, 0xfffffffff840001, 0xfffffffff6a0001, 0xfffffffff5a0001, 0xfffffffff2a0001,
           0xfffffffff240001, 0xffffffffefe0001, 0xffffffffeca0001, 0xffffffffe9e0001, 0xffffffffe7c0001,
           0xffffffffe740001, 0xffffffffe520001),
    "45": (0x1fffffc20001, 0x1fffff980001, 0x1fffff7e0001, 0x1fffff360001, 0x1fffff060001, 0x1ffffede0001,
           0x1ffffeca0001, 0x1ffffeb40001, 0x1ffffe760001, 0x1ffffe640001, 0x1ffffe520001, 0x1ffffe0c0001),
}
RING_SET = {8192: "60-40-60", 16384: "60-40-40-60", 32768: "60-45x4-60"}
RING_SCALE = {8192: 40, 16384: 40, 32768: 45, 65536: 40}


def _case(kind, N, primes=None, limbs=0, name=None, **more):
    c = {"kind": kind, "N": N, "primes": primes or RING_SET[N], "limbs": limbs}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A client with a handful of encrypted parameters (a small layer): one ciphertext, all latency.
        _case("encrypt", 8192, params=2500, name="encrypt-1ct-n8192"),
        # The smallest whole round: three clients, a model of 100,000 parameters, everything encrypted.
        _case("round", 8192, params=100_000, clients=3, ratio=1.0, name="round-3c-100k-full"),
        # ResNet-18-sized update, ten clients, everything encrypted: the ordinary full-encryption round.
        _case("round", 16384, params=11_700_000, clients=10, ratio=1.0, name="round-10c-11.7M-full"),
        # ResNet-50-sized update, ten clients, top 10 % encrypted, the rest averaged in plaintext.
        _case("round", 16384, params=25_600_000, clients=10, ratio=0.1, name="round-10c-25.6M-top10"),
        # BERT-base-sized update, eight clients, top 10 %, the long ring with six primes.
        _case("round", 32768, params=110_000_000, clients=8, ratio=0.1, name="round-8c-110M-top10"),
        # The same ResNet-50-sized round as a client program with host buffers calls it.
        _case("host", 16384, params=25_600_000, clients=10, ratio=0.1, name="host-10c-25.6M-top10"),
        # BERT-base-sized update, everything encrypted, from host buffers: the largest call there is.
        _case("host", 32768, params=110_000_000, clients=8, ratio=1.0, name="host-8c-110M-full"),
        # The server alone, with many small clients.
        _case("server", 8192, params=100_000, clients=64, name="server-64c-100k"),
        # The receiver alone: the decoded 1 % of a BERT-base-sized model, long ring.
        _case("open", 32768, params=1_100_000, name="open-1.1M-n32768"),
        # The mask of a ResNet-50-sized model, made anew when the sensitivity map changes.
        _case("mask", 16384, params=25_600_000, ratio=0.1, name="mask-25.6M-top10"),
        # Batched transforms at the ring of the ordinary round, and the largest ring with all twelve primes.
        _case("ntt", 16384, batch=256, name="ntt-n16384-b256"),
        _case("ntt", 65536, "60", 12, batch=61, name="ntt-n65536-l12-b61"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# ciphertexts that a drawn case may hold on the device
_MOST_BYTES = 8e9


def _most_params(N, limbs, clients):
    """Encrypted parameters whose ciphertexts, for all clients, stay within _MOST_BYTES (32 bytes per limb each)."""
    return int(_MOST_BYTES / (32 * limbs * clients))


def draw(rng):
    kind = rng.choice(["round", "round", "round", "encrypt", "encrypt", "server", "open", "host", "mask", "ntt", "ntt"])
    if kind == "ntt":
        N = rng.choice([8192, 16384, 32768, 65536])
        primes = rng.choice(["60", "45"] + ([RING_SET[N]] if N in RING_SET else []))
        limbs = rng.choice([2, 4, 8, 12]) if primes in ("60", "45") else len(SETS[primes])
        return _case("ntt", N, primes, limbs, batch=_log_int(rng, 1, min(4096, 2e9 / (8 * N * limbs))))
    if kind == "mask":
        return _case("mask", rng.choice([8192, 16384, 32768]), params=_log_int(rng, 1000, 60_000_000),
                     ratio=round(rng.uniform(0.005, 0.5), 4))
    if kind == "encrypt":
        N = rng.choice([8192, 16384, 32768, 65536])
        primes = RING_SET[N] if N in RING_SET and rng.random() < 0.6 else rng.choice(["60", "45"])
        limbs = rng.choice([2, 4, 8]) if primes in ("60", "45") else len(SETS[primes])
        return _case("encrypt", N, primes, limbs, params=_log_int(rng, 100, min(12_000_000, _most_params(N, limbs, 1))))
    N = rng.choice([8192, 16384, 32768])
    limbs = len(SETS[RING_SET[N]])
    if kind == "open":
        return _case("open", N, params=_log_int(rng, 1000, 12_000_000))
    if kind == "server":
        clients = rng.randint(2, 100)
        return _case("server", N, clients=clients, params=_log_int(rng, 1000, _most_params(N, limbs, clients)))
    clients = rng.randint(2, 12)
    ratio = rng.choice([1.0, 1.0, round(rng.uniform(0.005, 0.3), 4)])
    most = min(30_000_000, int(_most_params(N, limbs, clients) / ratio))
    return _case(kind, N, clients=clients, ratio=ratio, params=_log_int(rng, 1000, most))


# --------------------------------------------------------------------------- sizes of a case

def _primes(c):
    p = SETS[c["primes"]]
    return list(p[:c["limbs"]] if c["limbs"] else p)


def _encrypted(c):
    return c["params"] if c.get("ratio", 1.0) >= 1.0 else int(round(c["ratio"] * c["params"]))


def _cts(c):
    n = c["N"] // 2
    return (_encrypted(c) + n - 1) // n


# --------------------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _update(g, P):
    """A model update: normal with standard deviation 0.01."""
    return torch.randn(P, generator=g, device="cuda", dtype=torch.float32).mul_(0.01)


def _scores(g, P):
    """Sensitivity scores |gradient| * |weight|, both normal with standard deviation 0.02."""
    a = torch.randn(P, generator=g, device="cuda", dtype=torch.float32).mul_(0.02).abs_()
    return a.mul_(torch.randn(P, generator=g, device="cuda", dtype=torch.float32).mul_(0.02).abs_())


def _alpha(g, clients):
    """Normalised weights of the clients (dataset sizes)."""
    sizes = torch.randint(100, 1001, (clients,), generator=g, device="cuda").double()
    return (sizes / sizes.sum()).tolist()


def _residues(g, shape, primes):
    """Uniform residues modulo each prime, int64 [..., L, N]."""
    out = torch.empty(shape, dtype=torch.int64, device="cuda")
    for j, q in enumerate(primes):
        out[..., j, :].copy_(torch.randint(0, q, out[..., j, :].shape, generator=g, device="cuda"))
    return out


def prepare(case, seed):
    g = _generator(seed)
    kind, N, primes = case["kind"], case["N"], _primes(case)
    L = len(primes)
    s = {"case": case, "seed": seed}
    s["ctx"] = ctx = he.he_ctx_create(N, primes, RING_SCALE[N])
    if kind == "ntt":
        s["forward"] = _residues(g, (case["batch"], L, N), primes)
        s["inverse"] = _residues(g, (case["batch"], L, N), primes)
        return s
    P = case["params"]
    if kind == "mask":
        s["scores"] = _scores(g, P)
        return s
    T = _cts(case)
    if kind == "server":
        s["cts"] = [_residues(g, (T, 2, L, N), primes) for _ in range(case["clients"])]
        s["alpha"] = _alpha(g, case["clients"])
        s["agg"] = torch.empty((T, 2, L - 1, N), dtype=torch.int64, device="cuda")
        return s
    s["keys"] = he.he_keygen(ctx, seed * 2 + 1)
    he.he_ctx_reserve(ctx, T * (N // 2))
    if kind == "encrypt":
        s["x"] = _update(g, P)
        s["ct"] = torch.empty((T, 2, L, N), dtype=torch.int64, device="cuda")
        return s
    if kind == "open":
        # the aggregate of two encrypted updates
        cts = [he.he_encrypt(ctx, s["keys"], he.he_pack(ctx, None, _update(g, P))[0], seed, i) for i in range(2)]
        s["agg"] = he.he_weighted_aggregate(ctx, cts, [0.25, 0.75])
        return s
    clients, k = case["clients"], _encrypted(case)
    s["alpha"] = _alpha(g, clients)
    s["mask"] = he.he_select_mask(ctx, _scores(g, P), k) if k < P else None
    xs = [_update(g, P) for _ in range(clients)]
    if kind == "host":
        s["xs"] = []
        for x in xs:
            h = torch.empty(P, dtype=torch.float32, pin_memory=True)
            s["xs"].append(h.copy_(x))
        s["out"] = torch.empty(P, dtype=torch.float64, pin_memory=True)
        return s
    s["xs"] = xs
    s["cts"] = [torch.empty((T, 2, L, N), dtype=torch.int64, device="cuda") for _ in range(clients)]
    s["agg"] = torch.empty((T, 2, L - 1, N), dtype=torch.int64, device="cuda")
    s["z"] = torch.empty(T * (N // 2), dtype=torch.float64, device="cuda")
    s["out"] = torch.empty(P, dtype=torch.float64, device="cuda")
    return s


# --------------------------------------------------------------------------- one pass

def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "ntt":                       # in place, as the entry points work
        return [he.he_ntt_forward(ctx, s["forward"]), he.he_ntt_inverse(ctx, s["inverse"])]
    if kind == "mask":
        mask = he.he_select_mask(ctx, s["scores"], _encrypted(case))
        return he.he_mask_indices(mask)
    if kind == "server":
        return he.he_weighted_aggregate(ctx, s["cts"], s["alpha"], out=s["agg"])
    keys = s["keys"]
    if kind == "encrypt":
        sel, _ = he.he_pack(ctx, None, s["x"])
        return he.he_encrypt(ctx, keys, sel, s["seed"], 0, out=s["ct"])
    if kind == "open":
        z = he.he_decrypt(ctx, keys, s["agg"])
        return he.he_unpack(ctx, None, z, None, case["params"])
    if kind == "host":
        return he.he_round_host(ctx, keys, s["mask"], s["xs"], s["alpha"], s["seed"], s["out"])
    mask, rests = s["mask"], []
    for i, x in enumerate(s["xs"]):
        sel, rest = he.he_pack(ctx, mask, x)
        rests.append(rest)
        he.he_encrypt(ctx, keys, sel, s["seed"], i, out=s["cts"][i])
    he.he_weighted_aggregate(ctx, s["cts"], s["alpha"], out=s["agg"])
    avg = he.he_plain_aggregate(ctx, rests, s["alpha"]) if mask is not None else None
    z = he.he_decrypt(ctx, keys, s["agg"], out=s["z"])
    model = he.he_unpack(ctx, mask, z, avg, case["params"], out=s["out"])
    return {"model": model, "aggregate": s["agg"], "ciphertexts": s["cts"]}


# --------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    kind, N, L = case["kind"], case["N"], len(_primes(case))
    n = N // 2
    if kind == "ntt":                       # every word read and written once by either transform
        return {"bytes": 2 * 16.0 * case["batch"] * L * N, "flops": 2.0 * case["batch"] * L * (N // 2) * math.log2(N)}
    P = case["params"]
    if kind == "mask":                      # scores in, index list out
        return {"bytes": 4.0 * P + 4.0 * _encrypted(case), "flops": 0.0}
    T, k = _cts(case), _encrypted(case)
    ct, agg = 16.0 * L * N * T, 16.0 * (L - 1) * N * T
    slot = 5.0 * n * math.log2(n) * T       # one slot transform of every ciphertext index
    if kind == "encrypt":                   # the update in, the ciphertext out
        return {"bytes": 4.0 * P + ct, "flops": slot}
    if kind == "server":
        C = case["clients"]
        return {"bytes": C * ct + agg, "flops": 2.0 * C * 2 * L * N * T}
    if kind == "open":                      # limb 0 of both components in, the values out
        return {"bytes": 16.0 * N * T + 8.0 * P, "flops": slot}
    C = case["clients"]
    flops = (C + 1) * slot + 2.0 * C * (2 * L * N * T + P - k)
    if kind == "host":                      # updates in over PCIe, the model out; nothing else has to leave the chip
        return {"bytes": 4.0 * P * C + 8.0 * P, "flops": flops}
    # the calls of a round hand ciphertexts to one another: written by the clients, read by the server
    return {"bytes": 4.0 * P * C + 2 * C * ct + 2 * agg + 8.0 * P, "flops": flops}


def tolerance(case):
    """Masks, ciphertexts, aggregates and transforms are integers.  Decoded values are the slot transform, in fp64, of
    integers that are exact: a double-precision transform of 2^12 to 2^14 values against the same in extended
    precision differs by 2.5e-16 to 2.9e-16 (2-norm, relative; single values by up to 1.3e-15 of the rms); a weighted average of
    plaintext entries by less."""
    if case["kind"] in ("round", "host", "open"):
        return {"rel": 1e-15, "max": 1e-14}
    return "exact"
