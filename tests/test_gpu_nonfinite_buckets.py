"""Words and averages beside an infinity or a NaN.

A bucket that holds one has a norm that is not finite: the scale of its codes is 0, so every code of it is s
(dq.h), its averages are NaN, and nothing outside the bucket changes.  All routes agree: norms and codes in one
pass, codes for given norms, the whole round.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SEED = 0xBAD_F10A7
SEGS = [70, 4097, 31, 1, 3 * 4096 + 77, 64, 9000]
BAD = [np.nan, np.inf, -np.inf]


@pytest.fixture(scope="module")
def G(dqlib):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    import gpu_util
    return gpu_util


@pytest.mark.parametrize("b", [1, 2, 3, 4, 5, 7, 8, 11, 16])
@pytest.mark.parametrize("bucket,norm", [(32, 2), (96, 2), (512, 2), (2048, 2), (4096, 2), (1056, 2), (0, 2), (96, 0), (512, 0), (4096, 0)])
def test_a_bad_entry_stays_in_its_bucket(G, bucket, norm, b):
    dq = G.dq
    M = 3
    ref = oracle.Layout(SEGS, bucket if bucket else oracle.whole_tensor_bucket(SEGS))
    rng = np.random.default_rng(100 * bucket + b)
    g = np.full((M, ref.D32), np.nan, np.float32)                 # (padding, ignored)
    for o, n in zip(ref.offsets, SEGS):
        g[:, o: o + n] = rng.standard_normal((M, n)).astype(np.float32)
    clean = np.nan_to_num(g)
    hit = np.zeros((M, ref.nb), bool)
    where = [k for k in range(ref.nb) if k % 5 == 1] or [0]       # full and short buckets, one worker each
    for i, k in enumerate(where):
        at, n, m = int(ref.bucket_start[k]), int(ref.bucket_len[k]), i % M
        for j in range(1 + i % 3):
            g[m, at + int(rng.integers(0, n))] = BAD[(i + j) % 3]
        clean[m, at: at + n] = 0.0
        hit[m, k] = True
    dirty = np.zeros(ref.D32, bool)                               # elements whose average is NaN
    for k in np.flatnonzero(hit.any(axis=0)):
        dirty[int(ref.bucket_start[k]): int(ref.bucket_start[k]) + int(ref.bucket_len[k])] = b > 1
    r = G.GpuRound(SEGS, bucket, M, norm=norm)
    r.set_grads(g)
    r.set_b(b)
    norms = r.norms().copy()
    np.testing.assert_array_equal(np.isfinite(norms), ~hit)
    assert r.read_status() == dq.STAT_NONFINITE
    as_zero = np.where(hit, np.float32(0), norms)
    want = oracle.quantize_pack(ref, clean, as_zero, b, SEED, 2)
    avg = oracle.unpack_dequant_average(ref, want, as_zero, b)
    nw = ref.packed_words(b)

    def check(packed, out):
        np.testing.assert_array_equal(packed[:, :nw], want)
        if out is not None:
            np.testing.assert_array_equal(np.isnan(out), dirty)
            assert G.rel_l2(out[~dirty], avg[~dirty]) <= 1e-6

    packed = r.quantize(SEED, 2, fill=-1)                          # given norms
    out = r.average(fill=1.0).copy()
    check(packed, out)
    if bucket:
        check(r.norms_quantize(SEED, 2, fill=-1)[1], None)
    nbytes = dq.round_workspace_bytes(r.lay, M)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    for whole in (False, True):
        r.g_packed.view.fill_(-1)
        r.g_out.view.fill_(1.0)
        if whole:
            dq.norms_quantize_average(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 2, r.g_norms.view, r.g_packed.view, r.pstride,
                                      r.g_out.view, dq.Rule.fixed(b), ws, nbytes, r.status)
        else:
            dq.quantize_average(r.lay, r.grads, r.stride, M, r.g_norms.view, r.g_b.view, SEED, 2, r.g_packed.view, r.pstride,
                                r.g_out.view, r.status)
        one = r.g_out.view.cpu().numpy()
        check(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(M, -1), one)
        np.testing.assert_array_equal(one, out)                     # (NaN where the other is NaN)
    assert r.read_status() == dq.STAT_NONFINITE and r.guards_intact()
