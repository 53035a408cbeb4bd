"""The default key switch (one-hot digits times key limbs on the tensor pipe):
tile edges in gates, unaligned rows, and keys and digits at the ends of the
limbs' and sums' exact ranges.  Words mod 2^32: every comparison is for
equality."""
import numpy as np
import pytest

from conftest import oparams
from paper_2005_01945_gb300 import synth

pytestmark = pytest.mark.gpu
N, T, D = 1024, 8, 3


@pytest.fixture(scope="module")
def gpu(orc):
    import torch
    from paper_2005_01945_gb300 import api, build
    build.build()
    return dict(torch=torch, api=api, p=synth.TFHEParams())


def _ctx(gpu, ksk):
    api, p = gpu["api"], gpu["p"]
    ctx = api.Context(p)
    ctx.set_keys(api.to_device(np.zeros((p.n, 4, 2, N), dtype=np.uint32)), api.to_device(ksk))
    return ctx


def _run(gpu, ctx, big):
    torch, api = gpu["torch"], gpu["api"]
    out = torch.zeros((len(big), 512), dtype=torch.int32, device="cuda")
    ctx.keyswitch(big if torch.is_tensor(big) else api.to_device(big), out)
    torch.cuda.synchronize()
    assert ctx.status() == 0
    return out.cpu().numpy().view(np.uint32)


def test_gate_tile_edges(gpu, orc):
    torch, api, p = gpu["torch"], gpu["api"], gpu["p"]
    g = synth._gen(31, "kst")
    ksk = g.integers(0, 1 << 32, size=(N, T, D, p.n + 1), dtype=np.uint64).astype(np.uint32)
    ctx = _ctx(gpu, ksk)
    try:
        big = g.integers(0, 1 << 32, size=(1300, api.BIG_STRIDE), dtype=np.uint64).astype(np.uint32)
        want = orc.keyswitch(oparams(p), ksk, big[:, :N + 1])
        dev = api.to_device(big)
        for count in (1, 64, 65, 127, 128, 129, 255, 256, 257, 513, 1300):
            got = _run(gpu, ctx, dev[:count].contiguous())
            assert np.array_equal(got[:, :p.n + 1], want[:count])
            assert not got[:, p.n + 1:].any()
        # rows that do not start on 16 bytes
        flat = torch.zeros(300 * api.BIG_STRIDE + 1, dtype=torch.int32, device="cuda")
        odd = flat[1:].view(300, api.BIG_STRIDE)
        odd.copy_(dev[:300])
        assert np.array_equal(_run(gpu, ctx, odd)[:, :p.n + 1], want[:300])
    finally:
        ctx.close()


# all limbs at -1024 / -512, all at 1023 / 511, the wraps of the two lower limbs
@pytest.mark.parametrize("word", [(-1024 - (1024 << 11) - (511 << 22)) % (1 << 32),
                                  1023 + (1023 << 11) + (511 << 22), 1 << 31, (1 << 31) - 1,
                                  1024, 0xFFFFFBFF, 0xFFFFFFFF])
@pytest.mark.parametrize("count", [3, 70, 4000])
def test_extreme_limbs_and_sums(gpu, word, count):
    api, p = gpu["api"], gpu["p"]
    ctx = _ctx(gpu, np.full((N, T, D, p.n + 1), word, dtype=np.uint32))
    try:
        big = np.full((count, api.BIG_STRIDE), 0xFFFF0000, dtype=np.uint32)   # digits 3
        big[1] = 0x7FFF7FFF                   # digits 1 3 3 ..
        big[2] = 0xFFFFFFFF                   # rounds to digits 0
        got = _run(gpu, ctx, big)
        full = (0xFFFF0000 - 8192 * word) % (1 << 32)
        assert (got[0, :p.n] == (-8192 * word) % (1 << 32)).all() and got[0, p.n] == full
        assert (got[1, :p.n] == (-8192 * word) % (1 << 32)).all()
        assert not got[2, :p.n].any() and got[2, p.n] == 0xFFFFFFFF
        assert (got[3:] == got[0]).all()
    finally:
        ctx.close()


def test_context_without_limbs(gpu, orc):
    """Keys set while memory is too short for the key's limbs: the key switch
    and the autotuner run on the key's rows, before and after tuning."""
    torch, api, p = gpu["torch"], gpu["api"], gpu["p"]
    g = synth._gen(32, "nolimb")
    ksk = g.integers(0, 1 << 32, size=(N, T, D, p.n + 1), dtype=np.uint64).astype(np.uint32)
    big = g.integers(0, 1 << 32, size=(608, api.BIG_STRIDE), dtype=np.uint64).astype(np.uint32)
    want = orc.keyswitch(oparams(p), ksk, big[:, :N + 1])
    bk_dev = api.to_device(np.zeros((p.n, 4, 2, N), dtype=np.uint32))
    ksk_dev = api.to_device(ksk)
    limbs = N * T * D * 512 * 3 * 2
    ctx = api.Context(p)
    try:
        ctx.set_option(api.OPT_TEST_FREE_HBM, limbs - 1)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx.set_keys(bk_dev, ksk_dev)
        ctx.set_option(api.OPT_TEST_FREE_HBM, 0)
        # the transformed key and the padded rows alone
        assert before - torch.cuda.mem_get_info()[0] < p.n * 4 * 2 * 2 * N * 4 + limbs // 3 * 2 + limbs // 2
        assert np.array_equal(_run(gpu, ctx, big)[:, :p.n + 1], want)
        ctx.autotune()
        assert np.array_equal(_run(gpu, ctx, big)[:, :p.n + 1], want)
        # with room again, the limbs come with the next keys
        ctx.set_keys(bk_dev, ksk_dev)
        assert np.array_equal(_run(gpu, ctx, big)[:, :p.n + 1], want)
    finally:
        ctx.close()


@pytest.mark.parametrize("count", [65, 300])
def test_wait_timeout_is_reported_and_recoverable(gpu, orc, count):
    """The issuing thread's first wait runs out, and the waits of the
    warps that write the one-hot rows run out or are called off: the kernel ends,
    the status word says so (bit 2), and the next call is exact."""
    api, p, torch = gpu["api"], gpu["p"], gpu["torch"]
    g = synth._gen(33, "stall")
    ksk = g.integers(0, 1 << 32, size=(N, T, D, p.n + 1), dtype=np.uint64).astype(np.uint32)
    big = g.integers(0, 1 << 32, size=(count, api.BIG_STRIDE), dtype=np.uint64).astype(np.uint32)
    want = orc.keyswitch(oparams(p), ksk, big[:, :N + 1])
    ctx = _ctx(gpu, ksk)
    try:
        out = torch.zeros((count, 512), dtype=torch.int32, device="cuda")
        for _ in range(3):
            ctx.set_option(api.OPT_TEST_KS_STALL, 1)
            ctx.keyswitch(api.to_device(big), out)
            ctx.set_option(api.OPT_TEST_KS_STALL, 0)
            assert ctx.status() == 4
            assert np.array_equal(_run(gpu, ctx, big)[:, :p.n + 1], want)
    finally:
        ctx.close()


def test_beyond_65535_gate_tiles(gpu, orc):
    """More gate tiles than the smaller grid dimensions hold (65,535 x 256
    samples), around that edge and in the last, ragged tile."""
    torch, api, p = gpu["torch"], gpu["api"], gpu["p"]
    edge = 65535 * 256
    count = edge + 257
    if torch.cuda.mem_get_info()[0] < count * (api.BIG_STRIDE + 512) * 4 + (4 << 30):
        pytest.skip("needs 107 GB of free device memory")
    g = synth._gen(34, "many")
    ksk = g.integers(0, 1 << 32, size=(N, T, D, p.n + 1), dtype=np.uint64).astype(np.uint32)
    sample = np.array([0, 255, 256, edge - 1, edge, edge + 255, edge + 256])
    rows = g.integers(0, 1 << 32, size=(len(sample), api.BIG_STRIDE), dtype=np.uint64)
    rows = rows.astype(np.uint32)
    want = orc.keyswitch(oparams(p), ksk, np.ascontiguousarray(rows[:, :N + 1]))
    ctx = _ctx(gpu, ksk)
    try:
        big = torch.zeros((count, api.BIG_STRIDE), dtype=torch.int32, device="cuda")
        for s, r in zip(sample, rows):
            big[int(s)].copy_(api.to_device(r))
        out = torch.full((count, 512), 7, dtype=torch.int32, device="cuda")
        ctx.keyswitch(big, out)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        got = np.stack([out[int(s)].cpu().numpy() for s in sample]).view(np.uint32)
        assert np.array_equal(got[:, :p.n + 1], want)
        assert not got[:, p.n + 1:].any()
        assert not out[1:255].any() and not out[edge + 1:edge + 255].any()   # zero samples
    finally:
        big = out = None
        torch.cuda.empty_cache()
        ctx.close()
