"""Failure detection of the blind rotations without a GPU fault: with the test
hook the wait for one tensor-pipe product runs out after about a second (the
product itself completes).  The kernel ends, the status word reports it (bit 2),
and the next call on the same context equals the oracle."""
import numpy as np
import pytest

from conftest import oparams
from paper_2005_01945_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu(orc):
    import torch
    from paper_2005_01945_gb300 import api, build
    build.build()
    p = synth.TFHEParams(n=24)
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


# Shapes 1 and 8: the first step and later ones; 700 and 200 gates: two gates per slot.
# Shape 16: a product of a gate's second CTA, so that the first one's wait for residues
# runs out two steps later; of a gate with one step, behind which the first CTA ends by
# itself; of a cluster's second gate
@pytest.mark.parametrize("shape,count,where", [(1, 3, (1, 2, 24)), (1, 700, (1, 24, 25, 30)),
                                               (8, 3, (1, 2, 20)), (8, 200, (1, 30)),
                                               (16, 3, (1, 2, 3)), (16, 100, (1, 3, 77, 100))])
def test_timeout_is_reported_and_recoverable(gpu, orc, shape, count, where):
    torch, api, p, P, ctx = gpu["torch"], gpu["api"], gpu["p"], gpu["P"], gpu["ctx"]
    g = synth._gen(37, f"stall{shape}{count}")
    cts = g.integers(0, 1 << 32, size=(count, 512), dtype=np.uint64).astype(np.uint32)
    cts[:, :p.n] = cts[:, :p.n] & 0x7FFFFFFF | 1 << 22     # every step rotates
    cts[2, :p.n] = 0
    cts[2, 5] = 1 << 30                    # one step
    cts[:, p.n + 1:] = 0
    want = orc.bootstrap(P, gpu["bk"], gpu["ksk"], cts[:, :p.n + 1], mu=1 << 29)
    dev = api.to_device(cts)
    ctx.set_option(api.OPT_BR_GROUP, shape)
    try:
        for k in where:
            out = torch.zeros((count, 512), dtype=torch.int32, device="cuda")
            ctx.set_option(api.OPT_TEST_BR_STALL, k)
            ctx.bootstrap(dev, out, mu=1 << 29)
            ctx.set_option(api.OPT_TEST_BR_STALL, 0)
            assert ctx.status() == 4
            ctx.bootstrap(dev, out, mu=1 << 29)
            assert ctx.status() == 0
            assert np.array_equal(out.cpu().numpy().view(np.uint32)[:, :p.n + 1], want)
    finally:
        ctx.set_option(api.OPT_TEST_BR_STALL, 0)
        ctx.set_option(api.OPT_BR_GROUP, 0)
