"""The workloads this library is measured on: what a program that draws its
random numbers from it has the library do, through the public entry points
(Generator, Plan, battery.counts, Server), from a few thousand numbers to a
full device.

listed() names them, draw() makes more of the same ranges, prepare() builds
what a program keeps (handles, plans, buffers, an engine), run() is one pass
and work() what the pass cannot do without.  exact() gives the FP32 outputs
in 64 bits by plain numpy and torch, from the recurrences as published.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1101_1846_gb300 import battery, capi, workloads
from paper_1101_1846_gb300.generator import BatchItem, Generator, Plan
from paper_1101_1846_gb300.laned import carve, wave_elems
from paper_1101_1846_gb300.scheduler import Piece
from paper_1101_1846_gb300.serving import Server

KINDS = ("mwc", "xor128", "kiss", "mwc16x2", "xorshift8", "kiss_xor")
STATE_WORDS = {"mwc": 2, "xor128": 4, "kiss": 4, "mwc16x2": 2, "xorshift8": 8, "kiss_xor": 4}
# 32-bit shifts, logical operations, additions and multiply-adds of one step
# (the paper's n_ops)
STEP_OPS = {"mwc": 2, "xor128": 7, "kiss": 11, "mwc16x2": 10, "xorshift8": 18, "kiss_xor": 20}
PAIR_STREAMS = capi.RNG_MAX_STREAMS_MWC16


def has_mult(kind: str) -> bool:
    return kind not in ("xor128", "xorshift8")


def max_streams(kind: str) -> int:
    return PAIR_STREAMS if kind in ("mwc16x2", "kiss_xor") else 1 << 22


def listed() -> list[dict]:
    return [
        # a simulation step that asks for a few numbers per thread: launch and latency
        {"name": "small_call", "op": "generate", "kind": "kiss", "fmt": "f32",
         "streams": 4096, "rows": 16},
        # few streams, a long sequence of each (workloads.MWC_4K)
        {"name": "mwc_4096x4096", "op": "generate", "kind": "mwc", "fmt": "u32",
         "streams": 4096, "rows": 4096},
        # one stream per replica of a simulation, a number of replicas of no particular
        # divisibility, long sequences
        {"name": "few_odd_streams", "op": "generate", "kind": "kiss", "fmt": "f32",
         "streams": 1001, "rows": 16384},
        # the ordinary bulk fill (workloads.XOR_KISS_1M)
        {"name": "xor128_2^20x1024", "op": "generate", "kind": "xor128", "fmt": "f32",
         "streams": 1 << 20, "rows": 1024},
        # the largest: a full device (workloads.FULL_4M), 16 GiB a call
        {"name": "full_2^22x1024", "op": "generate", "kind": "kiss", "fmt": "u32",
         "streams": 1 << 22, "rows": 1024},
        # bulk fill with an odd row length: no row is aligned
        {"name": "ragged_(2^20-1)x256", "op": "generate", "kind": "mwc", "fmt": "f32",
         "streams": (1 << 20) - 1, "rows": 256},
        # the paper's own KISS at its full stream count (16- but not 32-byte rows)
        {"name": "paper_kiss_76636x4096", "op": "generate", "kind": "kiss_xor", "fmt": "u32",
         "streams": PAIR_STREAMS, "rows": 4096},
        # Monte Carlo in registers: nothing stored but one count per stream
        {"name": "inline_disc_2^22x1024", "op": "inline", "kind": "mwc", "consumer": "disc",
         "streams": 1 << 22, "rows": 1024},
        # a restart at an arbitrary point of every stream, then the first rows from there
        {"name": "jump_2^20", "op": "jump", "kind": "xor128", "streams": 1 << 20, "rows": 16,
         "bits": 48},
        # many generators of mixed kinds, sizes and formats in one launch
        # (workloads.batched_instances, pieces of at most 1024 rows)
        {"name": "batch_512_mixed", "op": "batch", "count": 512, "max_streams": 65536,
         "max_rows": 1024, "recipe": 1234},
        # the statistical battery over a generator's outputs
        {"name": "battery_65536x4096", "op": "battery", "kind": "kiss", "streams": 65536,
         "rows": 4096},
        # the serving engine: a burst of requests from many clients
        {"name": "serving_48_requests", "op": "serving", "clients": 64, "streams": 65536,
         "requests": 48, "max_bytes": 64 << 20, "recipe": 5},
    ]


def _log(rng, lo: int, hi: int) -> int:
    return int(math.floor(lo * math.exp(rng.random() * math.log(hi / lo))))


def _streams(rng, kind: str, lo: int, hi: int) -> int:
    """Half the time any count, else a multiple of 4, 8 or 32."""
    n = _log(rng, lo, min(hi, max_streams(kind)) + 1)
    if rng.random() < 0.5:
        m = rng.choice((4, 8, 32))
        n = max(n // m * m, m)
    return n


def draw(rng) -> dict:
    op = rng.choice(("generate",) * 5 + ("inline", "jump", "batch", "battery", "serving"))
    kind = rng.choice(KINDS)
    if op == "generate":
        n = _streams(rng, kind, 32, 1 << 22)
        rows = _log(rng, 16, min(16384, (1 << 30) // n) + 1)
        return {"op": op, "kind": kind, "fmt": rng.choice(("u32", "f32")), "streams": n,
                "rows": rows}
    if op == "inline":
        n = _streams(rng, kind, 64, 1 << 22)
        return {"op": op, "kind": kind, "consumer": rng.choice(("sum_u32", "sum_u24", "disc")),
                "streams": n, "rows": _log(rng, 64, min(8192, (1 << 31) // n) + 1)}
    if op == "jump":
        return {"op": op, "kind": kind, "streams": _streams(rng, kind, 256, 1 << 20),
                "rows": _log(rng, 1, 65), "bits": rng.randint(8, 63)}
    if op == "batch":
        return {"op": op, "count": _log(rng, 8, 513), "max_streams": _log(rng, 1024, 65537),
                "max_rows": _log(rng, 64, 1025), "recipe": rng.randrange(1 << 30)}
    if op == "battery":
        n = _streams(rng, kind, 64, 1 << 18)
        return {"op": op, "kind": kind, "streams": n,
                "rows": _log(rng, 512, min(8192, (1 << 28) // n) + 1)}
    return {"op": "serving", "clients": _log(rng, 4, 65), "streams": _log(rng, 1024, 65537),
            "requests": rng.randint(4, 60), "max_bytes": _log(rng, 1 << 16, 1 << 26),
            "recipe": rng.randrange(1 << 30)}


def _instances(case: dict) -> list[workloads.Instance]:
    return workloads.batched_instances(case["count"], case["recipe"],
                                       (32, case["max_streams"]), (16, case["max_rows"] + 1))


def _requests(case: dict) -> list[workloads.Request]:
    log = workloads.request_log(duration_s=1.0, n_clients=case["clients"],
                                hi_bytes=case["max_bytes"], seed=case["recipe"])
    return log[:case["requests"]]


def prepare(case: dict, seed: int) -> dict:
    """Handles, plans and output buffers: all of them are kept from call to call."""
    op = case["op"]
    if op == "batch":
        ins = _instances(case)
        rng = np.random.Generator(np.random.PCG64(seed))
        gens = [Generator(i.kind, i.n_streams, int(s))
                for i, s in zip(ins, rng.integers(0, 2**63, len(ins), dtype=np.int64))]
        wave = [Piece(k, 0, i.n_per_stream) for k, i in enumerate(ins)]
        n_streams = [i.n_streams for i in ins]
        buf = torch.zeros(wave_elems(wave, n_streams), dtype=torch.int32, device="cuda")
        items = [BatchItem(g, i.n_per_stream, o, i.fmt)
                 for g, i, o in zip(gens, ins, carve(buf, wave, n_streams))]
        return {"op": op, "plan": Plan(items), "gens": gens, "out": buf}
    if op == "serving":
        log = _requests(case)
        server = Server(capi.RNG_KISS, case["clients"], case["streams"], seed_base=seed,
                        budget_bytes=8 << 30, chunk_rows=1024, tick_bytes=8 << 30)
        return {"op": op, "server": server, "held": None,
                "clients": np.array([r.client for r in log], dtype=np.uint32),
                "sizes": np.array([r.n_samples for r in log], dtype=np.uint64),
                "fmts": np.array([r.fmt for r in log], dtype=np.int32)}
    n, rows = case["streams"], case["rows"]
    g = Generator(case["kind"], n, seed)
    if op == "battery":
        return {"op": op, "u": g.generate(rows, "u32"), "streams": n, "rows": rows}
    state = {"op": op, "gen": g, "rows": rows}
    if op == "inline":
        state["consumer"] = case["consumer"]
        state["out"] = torch.empty(n, dtype=torch.int64, device="cuda")
        return state
    state["fmt"] = case.get("fmt", "u32")
    state["out"] = torch.empty((rows, n), device="cuda", dtype=torch.float32
                               if state["fmt"] == "f32" else torch.int32)
    if op == "jump":
        state["k"] = int(np.random.Generator(np.random.PCG64(seed)).integers(
            1 << (case["bits"] - 1), 1 << case["bits"], dtype=np.int64))
    return state


class _Result:
    """A request's output where the engine left it; keeps the engine alive."""

    def __init__(self, server: Server, rid: int):
        ptr, n, fmt = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_int()
        capi.check(capi.lib().rng_server_result(server.h, rid, ctypes.byref(ptr),
                                                ctypes.byref(n), ctypes.byref(fmt), None, None),
                   "rng_server_result")
        self.server = server
        self.__cuda_array_interface__ = {
            "data": (ptr.value, False), "shape": (n.value,), "version": 2,
            "typestr": "<f4" if fmt.value == capi.RNG_F32 else "<i4"}


def run(state: dict):
    op = state["op"]
    if op == "generate":
        return state["gen"].generate(state["rows"], state["fmt"], out=state["out"])
    if op == "inline":
        return state["gen"].generate_reduce(state["rows"], state["consumer"], out=state["out"])
    if op == "jump":
        state["gen"].jump(state["k"])
        return state["gen"].generate(state["rows"], state["fmt"], out=state["out"])
    if op == "batch":
        state["plan"].launch()
        return state["out"]
    if op == "battery":
        return battery.counts(state["u"], state["streams"], state["rows"])
    # serving: the burst before has been used and goes back to the engine
    server = state["server"]
    if state["held"] is not None:
        torch.cuda.current_stream().synchronize()
        server.release_many(state["held"])
    ids = server.submit_many(state["clients"], state["sizes"], state["fmts"])
    server.drain()
    state["held"], _ = server.take_arrays()
    return [torch.as_tensor(_Result(server, int(i)), device="cuda") for i in ids]


def _stream_bytes(kind: str) -> int:
    """State read and written and multiplier read, per stream and call."""
    return 8 * STATE_WORDS[kind] + 4 * has_mult(kind)


def work(case: dict) -> dict:
    op = case["op"]
    if op == "batch":
        ins = _instances(case)
        kinds = [KINDS[i.kind] for i in ins]
        return {"bytes": sum(i.n_streams * (4 * i.n_per_stream + _stream_bytes(k))
                             for i, k in zip(ins, kinds)),
                "flops": sum(i.n_streams * i.n_per_stream * STEP_OPS[k]
                             for i, k in zip(ins, kinds))}
    if op == "serving":
        log = _requests(case)
        samples = sum(r.n_samples for r in log)
        clients = len({r.client for r in log})
        return {"bytes": 4 * samples + clients * case["streams"] * _stream_bytes("kiss"),
                "flops": samples * STEP_OPS["kiss"]}
    n, rows, kind = case["streams"], case["rows"], case["kind"]
    if op == "battery":
        return {"bytes": 4 * n * rows, "flops": 4 * n * rows}
    ops = STEP_OPS[kind] * n * rows
    if op == "inline":
        return {"bytes": n * (8 + _stream_bytes(kind)), "flops": ops + n * rows}
    return {"bytes": 4 * n * rows + n * _stream_bytes(kind) * (2 if op == "jump" else 1),
            "flops": ops}


# ---------------------------------------------------------------- 64 bits
def _draws(seed: int, n: int):
    """splitmix64 started at seed + s for stream s: a function that returns
    the next draw of every stream."""
    z = (np.uint64(seed) + np.arange(n, dtype=np.uint64)).astype(np.uint64)

    def nxt():
        nonlocal z
        z = z + np.uint64(0x9E3779B97F4A7C15)
        r = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        r = (r ^ (r >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return r ^ (r >> np.uint64(31))
    return nxt


def _is_prime(n: int) -> bool:
    d, r = n - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for b in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(b, d, n)
        if x in (1, n - 1):
            continue
        for _ in range(r - 1):
            x = x * x % n
            if x == n - 1:
                break
        else:
            return False
    return True


def _safe_multipliers(k: int, bits: int) -> np.ndarray:
    """The k largest a < 2^bits with a 2^bits - 1 a safe prime (fewer if
    there are fewer), by a sieve over the small primes, then Miller-Rabin."""
    small = [p for p in range(3, 2000) if all(p % q for q in range(2, math.isqrt(p) + 1))]
    found, hi = [], (1 << bits) - 1
    while len(found) < k and hi > 1:
        a = np.arange(hi, max(hi - (1 << 20), 1), -1, dtype=np.int64)
        for p in small:  # p divides a 2^shift - 1: composite, unless it is p itself
            r, hit = a % p, np.zeros(len(a), dtype=bool)
            for shift in (bits - 1, bits):
                divides = r == pow(pow(2, shift, p), -1, p)
                hit |= divides & ((a << shift) - 1 != p) if bits < 32 else divides
            a = a[~hit]
        for x in a.tolist():
            q = (x << (bits - 1)) - 1
            if _is_prime(q) and _is_prime(2 * q + 1):
                found.append(x)
                if len(found) == k:
                    break
        hi -= 1 << 20
    return np.array(found, dtype=np.uint64)


def _seeded(kind: str, n: int, seed: int):
    """(state words, multipliers) of every stream as numpy uint64 arrays."""
    nxt, lo, hi = _draws(seed, n), np.uint64(0xFFFFFFFF), np.uint64(32)
    if kind in ("xor128", "xorshift8"):
        r = [nxt() for _ in range(STATE_WORDS[kind] // 2)]
        return [w for x in r for w in (x & lo, x >> hi)], []
    if kind in ("mwc", "kiss"):
        a = _safe_multipliers(n, 32)
        r = nxt()
        words, mult = [r & lo, (r >> hi) % a], [a]
    else:
        table = _safe_multipliers(392, 16)
        i, j = np.triu_indices(len(table), 1)
        a1, a2 = table[i[:n]], table[j[:n]]
        r, m, s = nxt(), np.uint64(0xFFFF), np.uint64(16)
        words = [(r & m) | ((((r >> s) & m) % a1) << s),
                 ((r >> hi) & m) | (((r >> np.uint64(48)) % a2) << s)]
        mult = [a1, a2]
    if kind in ("kiss", "kiss_xor"):
        r = nxt()
        words += [r & lo, r >> hi]
    return words, mult


def exact(case: dict, seed: int):
    """FP32 outputs in 64 bits.  None for whole numbers and for what takes
    too long here: many base-2^32 multipliers, and very many steps."""
    if case["op"] != "generate" or case["fmt"] != "f32":
        return None
    kind, n, rows = case["kind"], case["streams"], case["rows"]
    if (kind in ("mwc", "kiss") and n > 4096) or rows > 16384:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    words, mult = _seeded(kind, n, seed)
    w = [torch.from_numpy(x.astype(np.int64)).to(dev) for x in words]
    a = [torch.from_numpy(x.astype(np.int64)).to(dev) for x in mult]
    M = 0xFFFFFFFF

    def mwc():  # Eq. 2-3, base 2^32; the product wraps as a 64-bit word
        t = a[0] * w[0] + w[1]
        w[0], w[1] = t & M, (t >> 32) & M
        return w[0]

    def pair():  # Eq. 2-3, base 2^16, twice
        for i in range(2):
            w[i] = a[i] * (w[i] & 0xFFFF) + (w[i] >> 16)
        return ((w[0] << 16) + w[1]) & M

    def xs32():  # Eq. 6
        y = w[2] ^ (w[2] << 13 & M)
        y = y ^ (y >> 17)
        w[2] = y ^ (y << 5 & M)
        return w[2]

    def lcg():  # Eq. 7
        w[3] = (69069 * w[3] + 1234567) & M
        return w[3]

    def xor128():
        t = w[0] ^ (w[0] << 11 & M)
        w.append(w[3] ^ (w[3] >> 19) ^ t ^ (t >> 8))
        w.pop(0)
        return w[3]

    def xs8():  # Eq. 5
        t = w[7] ^ (w[7] << 13 & M)
        t = t ^ (t << 9 & M)
        e = w[0] ^ (w[0] >> 7)
        e = e ^ (e << 24 & M)
        w.append(t ^ w[4] ^ (w[4] << 7 & M) ^ w[3] ^ (w[3] >> 3) ^ w[1] ^ (w[1] >> 10) ^ e)
        w.pop(0)
        return w[7]

    step = {"mwc": mwc, "xor128": xor128, "mwc16x2": pair, "xorshift8": xs8,
            "kiss": lambda: (mwc() + xs32() + lcg()) & M,
            "kiss_xor": lambda: ((pair() ^ lcg()) + xs32()) & M}[kind]
    out = torch.empty((rows, n), dtype=torch.float64, device=dev)
    for j in range(rows):
        out[j] = (step() >> 8).double() * 2.0 ** -24
    return out
