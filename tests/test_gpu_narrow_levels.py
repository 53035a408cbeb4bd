"""The blind-rotation shapes of narrow levels: one bootstrap on a CTA's 16
warps and one on a cluster of two CTAs, at the edges of the level widths that
take them, over several gates per CTA, and at the ends of their exact ranges.
All outputs are words fixed by the scheme: every comparison is for equality."""
import numpy as np
import pytest

from conftest import oparams
from paper_2005_01945_gb300 import synth
from test_gpu_first_pass import test_extreme_digits_bit_exact as _extreme_digits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prime", [0, 1])
@pytest.mark.parametrize("shape", [8, 16])
def test_extreme_digits(orc, prime, shape):
    for limb in range(3):
        _extreme_digits(orc, prime, limb, shape)


@pytest.fixture(scope="module")
def gpu(orc):
    import torch
    from paper_2005_01945_gb300 import api, build
    build.build()
    p = synth.TFHEParams(n=24)   # short rotations: the shapes differ per step
    kd = synth.key_draws(p, synth.MASTER_SEED)
    d = api.to_device
    bk, ksk = api.keygen(p, d(kd.s), d(kd.S), d(kd.bk_mask), d(kd.bk_noise), d(kd.ksk_mask),
                         d(kd.ksk_noise))
    P = oparams(p)
    ctx = api.Context(p)
    ctx.set_keys(bk, ksk)
    yield dict(torch=torch, api=api, p=p, P=P, ctx=ctx,
               bk=orc.keygen_bk(P, kd.s, kd.S, kd.bk_mask, kd.bk_noise),
               ksk=orc.keygen_ksk(P, kd.s, kd.S, kd.ksk_mask, kd.ksk_noise))
    ctx.close()


@pytest.mark.parametrize("shape,count", [(0, 1), (0, 76), (0, 77), (0, 152), (0, 153), (16, 229),
                                         (0, 609), (0, 684), (0, 685), (0, 760), (0, 761),
                                         (8, 459)])
def test_widths(gpu, orc, shape, count):
    torch, api, p, P = gpu["torch"], gpu["api"], gpu["p"], gpu["P"]
    g = synth._gen(29, f"narrow{shape}{count}")
    cts = g.integers(0, 1 << 32, size=(count, 512), dtype=np.uint64).astype(np.uint32)
    cts[:, p.n + 1:] = 0
    cts[::3, :5] = 0                       # steps without a rotation
    cts[1::4, 7] = 1 << 31                 # rotation by N
    out = torch.zeros((count, 512), dtype=torch.int32, device="cuda")
    gpu["ctx"].set_option(api.OPT_BR_GROUP, shape)
    try:
        gpu["ctx"].bootstrap(api.to_device(cts), out, mu=1 << 29)
        torch.cuda.synchronize()
    finally:
        gpu["ctx"].set_option(api.OPT_BR_GROUP, 0)
    assert gpu["ctx"].status() == 0
    want = orc.bootstrap(P, gpu["bk"], gpu["ksk"], cts[:, :p.n + 1], mu=1 << 29)
    assert np.array_equal(out.cpu().numpy().view(np.uint32)[:, :p.n + 1], want)
