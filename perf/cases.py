"""Performance cases: the calls a user of the library makes, over the sizes
they are made at.

Each case names one public entry point and its sizes.  One key set per
process (a program keeps one context), the default parameter set (LWE n = 500,
N = 1024, Bg = 2^10, l = 2, key switch t = 8 base 4), fresh encryptions of
uniform random bits per seed.  Every output is an array of 32-bit torus words
that the scheme fixes bit for bit, so there is no rounding to compare
against: ``exact`` has no value for any of them.
"""
from __future__ import annotations

import atexit
import functools
import math

import torch

from paper_2005_01945_gb300 import api, synth

PARAMS = synth.TFHEParams()
KEY_SEED = 20050194

# Bootstrapped gates of one pass of the largest listed case (64 16-bit
# multiplications); no drawn case exceeds it.
MOST_GATES = 64 * 648

# 32-bit integer operations of one bootstrap: n CMux steps of 12 1024-point
# number-theoretic transforms (5120 butterflies at 7, 1024 twiddles at 3),
# 4096 pointwise 4-term products at 12, 4096 digits at 8, 2048 lifts at 12.
OPS_PER_BOOTSTRAP = 500 * (12 * (5120 * 7 + 1024 * 3) + 4096 * 12 + 4096 * 8 + 2048 * 12)
BK_BYTES = 500 * 4 * 2 * 1024 * 4          # bootstrapping key, coefficient words
KSK_ROWS = 1024 * 8 * 3                    # key-switching key rows of 501 words
LWE_BYTES = 501 * 4
BIG_BYTES = 1025 * 4

# The request mix of a server: gates, 16- and 32-bit additions and
# multiplications.
MIX = ((api.GATE, 1), (api.ADD, 16), (api.ADD, 32), (api.MUL, 16), (api.MUL, 32))


def listed():
    return [
        # one gate, as an interactive program evaluates a condition
        {"name": "gate-1", "call": "gates", "count": 1},
        # eight gates with a fixed memory budget: the smallest batch of the
        # benchmark, through the allocation-free call
        {"name": "gates-8-noalloc", "call": "gates_noalloc", "count": 8},
        # one level of a mid-size circuit, not a multiple of anything
        {"name": "gates-301", "call": "gates", "count": 301},
        # a wide level: bitwise operations on a few thousand encrypted bits
        {"name": "gates-4099", "call": "gates", "count": 4099},
        # plain refresh of stored ciphertexts (no gate, one input)
        {"name": "refresh-700", "call": "bootstrap", "count": 700},
        # the key-switching stage alone, at one GPU-filling level
        {"name": "keyswitch-608", "call": "keyswitch", "count": 608},
        # three byte additions: a deep, narrow circuit (latency)
        {"name": "add-8x3", "call": "add", "width": 8, "batch": 3},
        # the benchmark's batch of 32-bit additions
        {"name": "add-32x256", "call": "add", "width": 32, "batch": 256},
        # the benchmark's batch of 16-bit multiplications
        {"name": "mul-16x64", "call": "mul", "width": 16, "batch": 64},
        # one 32-bit product through the shallow multiplier (latency)
        {"name": "dadda-32x1", "call": "dadda", "width": 32, "batch": 1},
        # encrypted matrix-vector product, ragged shape
        {"name": "matvec-6x5-16", "call": "matvec", "rows": 6, "cols": 5, "width": 16},
        # twelve requests of the server's mix, submitted together to the
        # serving loop
        {"name": "serve-12", "call": "serve", "requests": 12},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["gates", "gates", "gates_noalloc", "bootstrap", "keyswitch", "add", "add",
                       "mul", "dadda", "matvec", "serve"])
    if call in ("gates", "bootstrap", "keyswitch"):
        return {"call": call, "count": _log_int(rng, 1, 9001)}
    if call == "gates_noalloc":
        return {"call": call, "count": _log_int(rng, 1, api.NOALLOC_MAX_GATES)}
    if call == "serve":
        return {"call": call, "requests": rng.randint(2, 12)}
    if call == "matvec":
        while True:
            c = {"call": call, "rows": rng.randint(1, 8), "cols": rng.randint(2, 8),
                 "width": rng.randint(4, 16)}
            if _gates(c) <= MOST_GATES:
                return c
    width = {"add": rng.randint(4, 32), "mul": rng.randint(4, 24),
             "dadda": rng.randint(8, 32)}[call]
    one = _gates({"call": call, "width": width, "batch": 1})
    return {"call": call, "width": width,
            "batch": _log_int(rng, 1, max(1, min(256, MOST_GATES // one)))}


_KIND = {"add": api.ADD, "mul": api.MUL, "dadda": api.MUL_DADDA}


def _mix(requests):
    return [MIX[k % len(MIX)] for k in range(requests)]


def _gates(case):
    """Bootstrapped gates of one pass."""
    call = case["call"]
    if call in _KIND:
        return case["batch"] * api.circuit_info(_KIND[call], case["width"])[0]
    if call == "matvec":
        return api.circuit_info(api.MATVEC, case["width"], case["rows"], case["cols"])[0]
    if call == "serve":
        return sum(1 if k == api.GATE else api.circuit_info(k, w)[0]
                   for k, w in _mix(case["requests"]))
    return 0 if call == "keyswitch" else case["count"]


def _rows(case):
    """Ciphertexts read and written by one pass."""
    call = case["call"]
    if call in _KIND:
        return 3 * case["batch"] * case["width"]
    if call == "matvec":
        return case["width"] * (case["rows"] * case["cols"] + case["cols"] + case["rows"])
    if call == "serve":
        return sum(3 * w for _, w in _mix(case["requests"]))
    return {"bootstrap": 2, "keyswitch": 1}.get(call, 3) * case["count"]


def work(case):
    gates = _gates(case)
    ksk = KSK_ROWS * LWE_BYTES
    if case["call"] == "keyswitch":
        count = case["count"]
        # 3/4 of the 8192 base-4 digits of a sample select a row to subtract
        return {"bytes": ksk + count * (BIG_BYTES + LWE_BYTES), "flops": count * 6144 * 501}
    return {"bytes": BK_BYTES + ksk + _rows(case) * LWE_BYTES,
            "flops": gates * (OPS_PER_BOOTSTRAP + 6144 * 501)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _words(g, *shape):
    return torch.randint(-2 ** 31, 2 ** 31, shape, generator=g, device="cuda",
                         dtype=torch.int64).to(torch.int32)


def _noise(g, sigma, *shape):
    z = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.round(z * (sigma * 2.0 ** 32)).to(torch.int64).to(torch.int32)


def _bits(g, *shape):
    return torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.uint8)


@functools.lru_cache(maxsize=None)
def _keys():
    """(LWE key, bootstrapping key, key-switching key) on the device."""
    p, g = PARAMS, _gen(KEY_SEED)
    s = _bits(g, p.n).to(torch.int32)
    big_s = _bits(g, p.N).to(torch.int32)
    rows = 2 * p.l
    bk, ksk = api.keygen(p, s, big_s, _words(g, p.n, rows, p.N),
                         _noise(g, p.sigma_bk, p.n, rows, p.N),
                         _words(g, p.N, p.ks_t, p.ks_digits, p.n),
                         _noise(g, p.sigma_lwe, p.N, p.ks_t, p.ks_digits))
    return s, bk, ksk


@functools.lru_cache(maxsize=None)
def _context(serving=False):
    """The context a program keeps; the server runs on one of its own."""
    _, bk, ksk = _keys()
    ctx = api.Context(PARAMS)
    ctx.set_keys(bk, ksk)
    if serving:
        ctx.serve_start(8 << 30)
        atexit.register(ctx.serve_stop)
    return ctx


def _encrypt(g, *shape):
    p = PARAMS
    return api.encrypt_bits(p, _keys()[0], _words(g, *shape, p.n),
                            _noise(g, p.sigma_lwe, *shape), _bits(g, *shape))


def _out(*shape):
    return torch.zeros(shape + (api.LWE_STRIDE,), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    call, g = case["call"], _gen(seed)
    st = {"call": call, "ctx": _context(call == "serve")}
    if call in ("gates", "gates_noalloc", "bootstrap"):
        count = case["count"]
        st.update(a=_encrypt(g, count), b=_encrypt(g, count), out=_out(count),
                  ops=torch.randint(0, 6, (count,), generator=g, device="cuda",
                                    dtype=torch.uint8))
    elif call == "keyswitch":
        # extracted samples: uniform masks
        st.update(big=_words(g, case["count"], api.BIG_STRIDE), out=_out(case["count"]))
    elif call in _KIND:
        batch, width = case["batch"], case["width"]
        st.update(width=width, batch=batch, a=_encrypt(g, batch, width),
                  b=_encrypt(g, batch, width), out=_out(batch, width))
    elif call == "matvec":
        r, c, w = case["rows"], case["cols"], case["width"]
        st.update(width=w, a=_encrypt(g, r, c, w), b=_encrypt(g, c, w), out=_out(r, w))
    else:
        st["requests"] = [(k, w, _encrypt(g, w), _encrypt(g, w), _out(w))
                          for k, w in _mix(case["requests"])]
        # a single gate's request carries its opcode
        st["requests"] = [(k, api.NAND if k == api.GATE else w, a, b, o)
                          for k, w, a, b, o in st["requests"]]
    # the server's worker has a stream of its own: its inputs are complete
    # before a request is submitted
    torch.cuda.synchronize()
    return st


def run(st):
    ctx, call = st["ctx"], st["call"]
    if call == "gates":
        ctx.bootstrap_gates(st["ops"], st["a"], st["b"], st["out"])
    elif call == "gates_noalloc":
        ctx.bootstrap_gates_noalloc(st["ops"], st["a"], st["b"], st["out"])
    elif call == "bootstrap":
        ctx.bootstrap(st["a"], st["out"])
    elif call == "keyswitch":
        ctx.keyswitch(st["big"], st["out"])
    elif call == "add":
        ctx.add_n(st["width"], st["a"], st["b"], st["out"])
    elif call == "mul":
        ctx.mul_n(st["width"], st["a"], st["b"], st["out"])
    elif call == "dadda":
        ctx.run_jobs([dict(kind=api.MUL_DADDA, width=st["width"], batch=st["batch"], in0=st["a"],
                           in1=st["b"], out=st["out"])])
    elif call == "matvec":
        ctx.matvec(st["width"], st["a"], st["b"], st["out"])
    else:
        ids = [ctx.serve_submit(k, w, a, b, o) for k, w, a, b, o in st["requests"]]
        for rid in ids:
            ctx.serve_wait(rid)
        return [o for _, _, _, _, o in st["requests"]]
    return st["out"]


def exact(case, seed):
    """Every output is 32-bit words fixed by the scheme: nothing to round."""
    return None
