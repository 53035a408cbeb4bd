"""Key files hold the transformed bootstrapping key as residues in [0, q), as
files written before the device copy was centred do; a key that went through
a file runs every blind-rotation shape to the same words."""
import numpy as np
import pytest

from paper_2005_01945_gb300 import synth

pytestmark = pytest.mark.gpu
Q = (134215681, 134203393)


@pytest.mark.parametrize("shape", [1, 8, 16])
def test_file_residues_and_results(tmp_path, shape):
    import torch
    from paper_2005_01945_gb300 import api, build
    build.build()
    p = synth.TFHEParams(n=6)
    kd = synth.key_draws(p, synth.MASTER_SEED)
    d = api.to_device
    bk, ksk = api.keygen(p, d(kd.s), d(kd.S), d(kd.bk_mask), d(kd.bk_noise), d(kd.ksk_mask),
                         d(kd.ksk_noise))
    path = tmp_path / "keys.tfhegb"
    g = np.random.default_rng(3)
    cts = g.integers(0, 1 << 32, size=(9, 512), dtype=np.uint64).astype(np.uint32)
    outs = []
    for load in (False, True):
        ctx = api.Context(p)
        try:
            if load:
                ctx.load_keys(path)
            else:
                ctx.set_keys(bk, ksk)
                ctx.save_keys(path)
            ctx.set_option(api.OPT_BR_GROUP, shape)
            out = torch.zeros((9, 512), dtype=torch.int32, device="cuda")
            ctx.bootstrap(d(cts), out)
            torch.cuda.synchronize()
            assert ctx.status() == 0
            outs.append(out.cpu().numpy())
        finally:
            ctx.close()
    assert np.array_equal(outs[0], outs[1])
    raw = np.fromfile(path, dtype=np.uint8)
    words = p.n * 4 * 4 * 1024
    ksk_bytes = 1024 * 8 * 3 * 512 * 4
    b = raw[raw.size - ksk_bytes - 4 * words:raw.size - ksk_bytes].view(np.uint32).reshape(-1, 2, 4096)
    assert (b[:, 0] < Q[0]).all() and (b[:, 1] < Q[1]).all()
    assert (b > (1 << 26) + 1).mean() > 0.4      # the upper half of [0, q) is there
