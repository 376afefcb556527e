"""Rounds in which a CTA takes its tiles through the workers together, against the separate calls, bit for bit.

Sizes around the edges of that kernel: one row, a tile and its neighbours, two tiles of a bucket of 2048, more
positions than CTAs, chunks of four (two) workers with and without a remainder, every width of a code (those that leave
from registers and those that go through shared memory), strides, an output that is only 16-byte aligned, buckets
that are zero, tiny or not finite.  The layouts of 3.3 million elements have too many tiles for it: the same comparison
for the kernel that takes those.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SEED = 0xC7A_711E5
RAGGED = [70, 1, 1023, 1024, 1025, 0, 4097, 31, 2048, 3 * 4096 + 77, 32, 9000]


@pytest.fixture(scope="module")
def G(dqlib):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    import gpu_util
    return gpu_util


CASES = [([d], bucket, M, b) for d, bucket, M, b in (
    (1, 32, 2, 4), (31, 512, 5, 8), (33, 1024, 4, 2), (1024, 512, 3, 16), (1025, 1024, 8, 4), (2047, 2048, 3, 5), (2048, 2048, 2, 4),
    (2080, 2048, 9, 6), (8193, 128, 17, 3), (70001, 512, 4, 8), (70001, 96, 6, 4), (70001, 0, 5, 4), (70001, 2048, 7, 8),
    (760001, 512, 3, 4), (2700001, 512, 2, 4), (1300001, 480, 2, 5), (1000001, 0, 2, 6), (1050001, 2048, 4, 4))]
CASES += [(RAGGED, bucket, 6, b) for bucket, b in ((32, 6), (96, 5), (480, 8), (512, 9), (2048, 7), (0, 11))]
CASES += [(RAGGED, 512, 5, b) for b in range(1, 17)] + [(RAGGED, 2048, 5, b) for b in range(1, 17)]
CASES += [(RAGGED + [3300000], bucket, 3, b) for bucket, b in ((32, 4), (96, 4), (480, 6), (512, 8), (2048, 4), (0, 3))]
CASES += [(RAGGED + [3300000], 4096, 3, 5), ([40] * 1100, 64, 5, 7)]
CASES = [c + (False,) for c in CASES] + [c + (True,) for c in CASES if c[3] in (4, 5, 8)]


@pytest.mark.parametrize("segs,bucket,M,b,linf", CASES)
def test_equals_the_separate_calls(G, segs, bucket, M, b, linf):
    dq = G.dq
    ref = oracle.Layout(segs, bucket if bucket else oracle.whole_tensor_bucket(segs))
    r = G.GpuRound(segs, bucket, M, stride=ref.D32 + 32 * (b % 3), norm=dq.NORM_LINF if linf else dq.NORM_L2)
    gen = torch.Generator(device="cuda").manual_seed(M * 100 + b)
    g = torch.full((M, r.stride), float("nan"), device="cuda")
    for i, (o, n) in enumerate(zip(ref.offsets.tolist(), segs)):
        g[:, o: o + n] = torch.randn((M, n), generator=gen, device="cuda") * 10.0 ** (i % 5 - 2)
    if len(segs) > 8:
        g[:, ref.offsets[8]: ref.offsets[8] + segs[8]] = 0.0
        g[0, ref.offsets[4]: ref.offsets[4] + segs[4]] *= 1e-30
    nonfinite = len(segs) > 8 and b % 2 == 0
    if nonfinite:
        g[M - 1, ref.offsets[3]] = float("inf")
    r.grads = g
    r.set_b(b)
    norms = r.norms().copy()
    packed = r.quantize(SEED, 9, fill=-1).copy()
    avg = r.average(fill=1.0).copy()
    x0 = np.linspace(-1, 1, r.lay.D32, dtype=np.float32)
    upd = r.update(0.125, x0).copy()
    nbytes = dq.round_workspace_bytes(r.lay, M)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    shifted = torch.empty(r.lay.D32 + 8, device="cuda")[4: 4 + r.lay.D32]          # 16-byte aligned, and no more
    for lr, want, out in ((None, avg, r.g_out.view), (0.125, upd, r.g_out.view), (None, avg, shifted), (0.125, upd, shifted)):
        r.set_b(b)
        r.g_packed.view.fill_(-1)
        r.g_norms.view.fill_(-1.0)
        out.copy_(torch.from_numpy(x0))
        dq.norms_quantize_average(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 9, r.g_norms.view, r.g_packed.view, r.pstride, out,
                                  dq.Rule.fixed(7), ws, nbytes, r.status, lr=lr)
        np.testing.assert_array_equal(r.g_norms.view.cpu().numpy().reshape(M, -1), norms)
        np.testing.assert_array_equal(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(M, -1), packed)
        np.testing.assert_array_equal(out.cpu().numpy(), want)
        assert r.g_b.view.tolist() == [7, 63]
    assert r.read_status() == (dq.STAT_NONFINITE if nonfinite else 0) and r.guards_intact()


@pytest.mark.parametrize("bucket,d", [(512, 70001), (2048, 70001), (480, 9000)])
def test_one_buffer_for_all_workers(G, bucket, d):
    """Stride 0: all workers read the same gradient, each with draws of its own."""
    dq = G.dq
    M, b = 6, 4
    r = G.GpuRound([d], bucket, M)
    g = torch.randn(r.lay.D32, device="cuda")
    r.grads, r.stride = g, 0
    r.set_b(b)
    r.norms()
    packed = r.quantize(SEED, 2, fill=-1).copy()
    avg = r.average().copy()
    nbytes = dq.round_workspace_bytes(r.lay, M)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    for whole in (False, True):
        r.g_packed.view.fill_(-1)
        if whole:
            dq.norms_quantize_average(r.lay, g, 0, M, r.g_b.view, SEED, 2, r.g_norms.view, r.g_packed.view, r.pstride, r.g_out.view,
                                      dq.Rule.fixed(3), ws, nbytes, r.status)
        else:
            dq.quantize_average(r.lay, g, 0, M, r.g_norms.view, r.g_b.view, SEED, 2, r.g_packed.view, r.pstride, r.g_out.view, r.status)
        np.testing.assert_array_equal(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(M, -1), packed)
        np.testing.assert_array_equal(r.g_out.view.cpu().numpy(), avg)
    assert r.read_status() == 0 and r.guards_intact()
