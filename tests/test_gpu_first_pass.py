"""The tensor-pipe first pass of the blind rotation's forward transforms at
the extremes of its exact range.

A two-step bootstrapping key drives the digits: the first CMux step (rotation
by 1 of a constant test vector, one digit of -1) sets the accumulator to any
chosen pair of polynomials, and the second (rotation by N, X^N P - P = -2P)
decomposes them into chosen digits.  They are -512 / 511 by the signs of the
constant operand's column of largest absolute sum, for each prime and limb,
so that column's fp32 sums reach the ends of their range; every output word
equals the oracle's schoolbook products."""
import numpy as np
import pytest

from paper_2005_01945_gb300 import synth

pytestmark = pytest.mark.gpu
Q = (134215681, 134203393)
N = 1024


def _limbs(q):
    """Balanced base-512 limbs [k1][i2][3] of the centred psi^(32 (2 k1 + 1) i2)."""
    psi = next(r for r in (pow(x, (q - 1) // (2 * N), q) for x in range(2, 1000))
               if pow(r, N, q) == q - 1)
    out = np.zeros((32, 32, 3), dtype=np.int64)
    for k1 in range(32):
        for i2 in range(32):
            v = pow(psi, 32 * (2 * k1 + 1) * i2, q)
            v -= q if v > q // 2 else 0
            for limb in range(2):
                d = (v + 256) % 512 - 256
                out[k1, i2, limb] = d
                v = (v - d) // 512
            out[k1, i2, 2] = v
    return out


@pytest.mark.parametrize("prime", [0, 1])
@pytest.mark.parametrize("limb", [0, 1, 2])
@pytest.mark.parametrize("shape", [1, 0])
def test_extreme_digits_bit_exact(orc, prime, limb, shape):
    import torch
    from paper_2005_01945_gb300 import api, build
    build.build()
    p = synth.TFHEParams(n=2)
    P = orc.Params(p.n, p.N, p.l, p.bg_bit, p.ks_t, p.ks_basebit)
    col = _limbs(Q[prime])[:, :, limb]
    col = col[np.abs(col).sum(axis=1).argmax()]            # largest |sum|, over i2
    d = np.where(np.repeat(col, 32) > 0, -512, 511)        # coefficient i1 + 32 i2
    mu = 1 << 21
    g = synth._gen(17, f"ext{prime}{limb}")
    bk = g.integers(0, 1 << 32, size=(p.n, 4, 2, N), dtype=np.uint64).astype(np.uint32)
    # digits d at both levels of the first polynomial, the opposite ends at
    # the second: -2P = d 2^22 + d' 2^12
    poly = [(-(a * (1 << 21) + b * (1 << 11))) % (1 << 32) for a, b in ((d, d), (-1 - d, d))]
    bk[0, 2, 0] = (-poly[0]) % (1 << 32)
    bk[0, 2, 1] = (mu - poly[1]) % (1 << 32)
    ksk = g.integers(0, 1 << 32, size=(N, p.ks_t, p.ks_digits, p.n + 1),
                     dtype=np.uint64).astype(np.uint32)
    cts = np.zeros((5, 512), dtype=np.uint32)
    cts[:, 0] = 1 << 21                                    # rotation by 1
    cts[:, 1] = np.array([N, N, 1, 2 * N - 1, 37], dtype=np.uint32) << 21
    ctx = api.Context(p)
    try:
        ctx.set_option(api.OPT_BR_GROUP, shape)
        ctx.set_keys(api.to_device(bk), api.to_device(ksk))
        out = torch.zeros((5, 512), dtype=torch.int32, device="cuda")
        ctx.bootstrap(api.to_device(cts), out, mu=mu)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        want = orc.bootstrap(P, bk, ksk, cts[:, :p.n + 1], mu=mu)
        assert np.array_equal(out.cpu().numpy().view(np.uint32)[:, :p.n + 1], want)
    finally:
        ctx.close()
