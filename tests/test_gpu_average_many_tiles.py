"""The average where every warp has several tiles of the layout: words and norms of the next tile on their way while
one is summed, the next tile's bucket and length, the parity of the tile of x.

(Layouts and worker counts are such that a whole round takes one kernel, which the test checks.)

Norms differ by up to 2^40 from bucket to bucket, so a word or a norm of another tile, worker or bucket is far out of
the bound: a value is a sum of M products level * scale, each with two roundings in its scale, added with M fused
roundings, so it lies within (M + 3) * 2^-24 of the sum of the magnitudes, which is at most the mean of the bucket's
norms over the workers.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SEED = 0xA7E_2A6E
# 6.7M elements: two tiles of 1024 and most of a third for each of the 2368 warps of a launch, which also is where a
# whole round takes one kernel
SEGS = [2_100_003, 70, 1_200_001, 4097, 0, 31, 2_200_000, 33, 1_200_033]


@pytest.fixture(scope="module")
def G(dqlib):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    import gpu_util
    oracle.set_threads(8)
    yield gpu_util
    oracle.set_threads(1)


@pytest.mark.parametrize("huge", [False, True])
@pytest.mark.parametrize("M,b,bucket", [(20, 2, 512), (24, 3, 512), (33, 4, 512), (20, 4, 480), (24, 2, 4096), (32, 3, 512), (33, 3, 0), (7, 4, 512),
                                        (20, 5, 480), (17, 6, 512), (21, 7, 512), (11, 7, 512), (12, 8, 512), (5, 16, 128)])
def test_every_element_of_every_tile(G, M, b, bucket, huge):
    dq = G.dq
    ref = oracle.Layout(SEGS, bucket if bucket else oracle.whole_tensor_bucket(SEGS))
    rng = np.random.default_rng(M * 100 + b)
    r = G.GpuRound(SEGS, bucket, M)
    # one exponent per bucket; `huge`: some beyond what the shifted sums hold, which ends a warp's fast loop midway
    expo = rng.integers(-20, 21, ref.nb)
    if huge:
        expo[rng.integers(0, ref.nb, max(1, ref.nb // 1500))] = 115
    bucket_of = np.full(ref.D32, -1, np.int32)
    for k in range(ref.nb):
        bucket_of[int(ref.bucket_start[k]): int(ref.bucket_start[k]) + int(ref.bucket_len[k])] = k
    valid = bucket_of >= 0
    of = torch.from_numpy(np.where(valid, bucket_of, 0)).cuda()
    scale = torch.from_numpy(np.ldexp(1.0, expo).astype(np.float32)).cuda()[of]
    gen = torch.Generator(device="cuda").manual_seed(M + b)
    r.grads = torch.randn((M, r.stride), generator=gen, device="cuda").mul_(scale)
    r.set_b(b)
    norms = r.norms().copy()
    packed = r.quantize(SEED, 3, fill=-1).copy()
    out = r.average(fill=1e30).copy()
    want = oracle.unpack_dequant_average(ref, packed[:, : ref.packed_words(b)], norms, b).astype(np.float64)
    bound = (M + 3) * 2.0 ** -24 * norms.astype(np.float64).mean(axis=0)
    assert np.all(out[~valid] == 0)
    assert np.all(np.abs(out - want)[valid] <= bound[bucket_of[valid]])
    x0 = np.linspace(-1, 1, ref.D32, dtype=np.float32)
    upd = r.update(0.25, x0).copy()
    # (one more rounding, of the result)
    moved = x0.astype(np.float64) - 0.25 * want
    assert np.all(np.abs(upd - moved)[valid] <= 0.25 * bound[bucket_of[valid]] + 2.0 ** -24 * np.abs(moved[valid]))
    np.testing.assert_array_equal(upd[~valid], x0[~valid])
    # and the kernel that never reads the words back, bit for bit
    nbytes = dq.round_workspace_bytes(r.lay, M)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    for lr, w in ((None, out), (0.25, upd)):
        r.set_b(b)
        r.g_out.view.copy_(torch.from_numpy(x0))
        dq.norms_quantize_average(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 3, r.g_norms.view, r.g_packed.view, r.pstride,
                                  r.g_out.view, dq.Rule.fixed(b), ws, nbytes, r.status, lr=lr)
        assert int(ws[128:132].view(torch.int32).item()) == 0, "two kernels: the average was compared with itself"
        np.testing.assert_array_equal(r.g_out.view.cpu().numpy(), w)
    assert r.read_status() == 0 and r.guards_intact()
