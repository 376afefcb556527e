"""``dq_norms_quantize_average`` and ``dq_quantize_average`` against the calls they merge.

Words, norms and the average (or the updated parameters) of the one-pass kernels equal those of
dq_norms_quantize_pack / dq_bucket_norms / dq_tensor_norms, dq_quantize_pack and
dq_unpack_dequant_average / dq_unpack_average_update bit for bit: same operations, same order over
the workers.  The next b is the rule's (threshold search on sums that differ by 1e-15).
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SEED = 0x0DD_5EED_71
# tensors shorter than a bucket, on and beside the edges of groups and warp tiles, an empty one
RAGGED = [70, 1, 1023, 1024, 1025, 0, 4097, 31, 2048, 3 * 4096 + 77, 32, 9000]


@pytest.fixture(scope="module")
def G(dqlib):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    import gpu_util
    return gpu_util


def _grads(ref, segs, M, seed):
    """Normal values of very different scales, a tensor of zeros, a bucket of tiny entries, NaN in the padding."""
    rng = np.random.default_rng(seed)
    g = np.full((M, ref.D32), np.nan, np.float32)
    for i, (o, n) in enumerate(zip(ref.offsets, segs)):
        g[:, o: o + n] = rng.standard_normal((M, n)).astype(np.float32) * np.float32(10.0 ** (i % 5 - 2))
    if len(segs) > 8:
        g[:, ref.offsets[8]: ref.offsets[8] + segs[8]] = 0.0
        g[0, ref.offsets[4]: ref.offsets[4] + segs[4]] *= np.float32(1e-30)
    return g


CASES = [(RAGGED, 512, 3, 4), (RAGGED, 32, 2, 7), (RAGGED, 1024, 5, 3), (RAGGED, 2048, 3, 5), (RAGGED, 4096, 2, 8),
         (RAGGED, 96, 2, 6), (RAGGED, 0, 3, 4),
         (RAGGED, 96, 3, 4), (RAGGED, 160, 2, 5), (RAGGED, 480, 3, 4), (RAGGED, 992, 2, 7), (RAGGED, 1056, 2, 4), ([100001], 96, 5, 3),
         ([1 << 18], 512, 4, 2), ([70001], 128, 1, 16), ([1], 4096, 2, 4),
         ([33] * 1100, 64, 2, 12), ([300000], 2048, 33, 4), (RAGGED, 512, 24, 5), (RAGGED, 4096, 24, 4), (RAGGED, 0, 24, 7), (RAGGED, 480, 24, 3),
         ([3 << 20], 512, 8, 4)] + [(RAGGED, 256, 2, b) for b in range(1, 17)]


@pytest.mark.parametrize("segs,bucket,M,b", CASES)
def test_one_call_equals_the_calls_it_merges(G, segs, bucket, M, b):
    dq = G.dq
    for norm in ((dq.NORM_L2, dq.NORM_LINF) if b in (4, 5) else (dq.NORM_L2,)):
        r = G.GpuRound(segs, bucket, M, norm=norm, packed_stride=None)
        ref = oracle.Layout(segs, bucket if bucket else oracle.whole_tensor_bucket(segs))
        g = _grads(ref, segs, M, 17 * M + b)
        r.set_grads(g)
        r.set_b(b)
        rule = dq.Rule.dynamic(10, 3, 0.37 * 10 * max(1e-30, float(np.nansum(g.astype(np.float64) ** 2)) / M) / 400.0, 0.9)
        # the separate calls
        norms = r.norms().copy()
        packed = r.quantize(SEED, 5, fill=-1).copy()
        avg = r.average(fill=1.0).copy()
        x0 = np.linspace(-1, 1, r.lay.D32, dtype=np.float32)
        upd = r.update(0.125, x0).copy()
        want_b = r.bits(rule)
        # one call with the norms given, one with everything; the average and the update; two runs in a row
        nbytes = dq.round_workspace_bytes(r.lay, M)
        ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        for whole in (False, True, True):
            for lr, want in ((None, avg), (0.125, upd)):
                r.set_b(b)
                r.g_packed.view.fill_(-1)
                r.g_out.view.copy_(torch.from_numpy(x0))
                if whole:
                    r.g_norms.view.fill_(-1.0)
                    dq.norms_quantize_average(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 5, r.g_norms.view, r.g_packed.view,
                                              r.pstride, r.g_out.view, rule, ws, nbytes, r.status, lr=lr)
                    assert tuple(r.g_b.view.cpu().tolist()) == want_b
                else:
                    dq.quantize_average(r.lay, r.grads, r.stride, M, r.g_norms.view, r.g_b.view, SEED, 5, r.g_packed.view,
                                        r.pstride, r.g_out.view, r.status, lr=lr)
                np.testing.assert_array_equal(r.g_norms.view.cpu().numpy().reshape(M, -1), norms)
                np.testing.assert_array_equal(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(M, -1), packed)
                np.testing.assert_array_equal(r.g_out.view.cpu().numpy(), want)
        assert r.read_status() == 0 and r.guards_intact()
        nw = ref.packed_words(b)
        np.testing.assert_array_equal(packed[:, :nw], oracle.quantize_pack(ref, np.nan_to_num(g), norms, b, SEED, 5))


def test_lost_first_wait_and_bad_bits(G):
    """A lost wait raises DQ_STAT_WAIT and nothing else; a b outside 1..16 writes no output but still gets its successor."""
    dq = G.dq
    for bucket, M in ((512, 3), (4096, 3), (96, 3), (512, 40), (4096, 40), (96, 40)):        # one kernel; codes, then average
        r = G.GpuRound(RAGGED, bucket, M)
        ref = oracle.Layout(RAGGED, bucket)
        r.set_grads(np.nan_to_num(_grads(ref, RAGGED, M, 1)))
        nbytes = dq.round_workspace_bytes(r.lay, M)
        ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")

        def call():
            dq.norms_quantize_average(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 0, r.g_norms.view, r.g_packed.view, r.pstride,
                                      r.g_out.view, dq.Rule.fixed(6), ws, nbytes, r.status)
            torch.cuda.synchronize()
        r.set_b(4)
        try:
            dq.debug_set_wait_limits(50_000_000, True)
            call()
        finally:
            dq.debug_set_wait_limits()
        assert r.read_status() == dq.STAT_WAIT and r.guards_intact()
        r.clear_status()
        r.g_packed.view.fill_(-7)
        r.set_b(17)
        call()
        assert r.read_status() == dq.STAT_BAD_BITS and bool((r.g_packed.view == -7).all())
        assert r.g_b.view.tolist() == [6, 31]
        r.clear_status()
        call()
        assert r.read_status() == 0 and r.guards_intact() and not bool((r.g_packed.view == -7).all())


@pytest.mark.parametrize("bucket,b", [(480, 4), (512, 4), (2048, 5), (512, 7)])
def test_repeated_passes_write_the_same_bits(G, bucket, b):
    """A stage is refilled while its warp may still be reading it unless the two are ordered: passes over
    two sets of gradients in turn, without a pause, give the same words and averages every time."""
    dq = G.dq
    d, M = (1 << 21) + 77, 8
    sets = []
    for i in range(2):
        r = G.GpuRound([d, 50001], bucket, M)
        gen = torch.Generator(device="cuda").manual_seed(i)
        r.grads = torch.randn((M, r.stride), generator=gen, device="cuda")
        r.set_b(b)
        r.norms()
        sets.append(r)

    def one(r):
        dq.quantize_average(r.lay, r.grads, r.stride, M, r.g_norms.view, r.g_b.view, SEED, 5, r.g_packed.view, r.pstride,
                            r.g_out.view, r.status)
        dq.norms_quantize_pack(r.lay, r.grads, r.stride, M, r.g_b.view, SEED, 5, r.g_norms.view, r.g_packed.view, r.pstride,
                               r.status)
    want = []
    for r in sets:
        r.g_packed.view.fill_(-1)
        r.quantize(SEED, 5)
        r.average()
        want.append((r.g_packed.view.clone(), r.g_out.view.clone(), r.g_norms.view.clone()))
    for _ in range(12):
        for r in sets:
            one(r)
        for r, (w, o, n) in zip(sets, want):
            assert torch.equal(r.g_packed.view, w) and torch.equal(r.g_out.view, o) and torch.equal(r.g_norms.view, n)
    assert all(r.read_status() == 0 and r.guards_intact() for r in sets)


@pytest.mark.parametrize("n_seg", [2, 31, 32, 33, 64, 500, 1023, 1100])
@pytest.mark.parametrize("bucket", [32, 512, 2048, 96])
def test_many_tensors_of_every_size(G, n_seg, bucket):
    """The warp-wide search of the tensor table (32 entries a step; 1023 tensors in shared memory, more from
    global memory): tables around its step sizes, empty tensors among them."""
    rng = np.random.default_rng(n_seg * 7 + bucket)
    segs = [int(x) for x in rng.choice([0, 1, 31, 33, 500, 2049, 5000], size=n_seg)]
    segs[0], segs[-1] = 4097, 70
    M, b = 2, 3
    ref = oracle.Layout(segs, bucket)
    g = np.zeros((M, ref.D32), np.float32)
    for o, n in zip(ref.offsets, segs):
        g[:, o: o + n] = rng.standard_normal((M, n)).astype(np.float32)
    r = G.GpuRound(segs, bucket, M)
    r.set_grads(g)
    r.set_b(b)
    norms, packed = r.norms_quantize(SEED, 1, fill=-1)
    nw = ref.packed_words(b)
    np.testing.assert_allclose(norms, oracle.bucket_norms(ref, g), rtol=1e-6)
    np.testing.assert_array_equal(packed[:, :nw], oracle.quantize_pack(ref, g, norms, b, SEED, 1))
    avg = r.average(fill=1.0).copy()
    r.g_packed.view.fill_(-1)
    G.dq.quantize_average(r.lay, r.grads, r.stride, M, r.g_norms.view, r.g_b.view, SEED, 1, r.g_packed.view, r.pstride,
                          r.g_out.view, r.status)
    np.testing.assert_array_equal(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(M, -1), packed)
    np.testing.assert_array_equal(r.g_out.view.cpu().numpy(), avg)
    assert r.read_status() == 0 and r.guards_intact()


@pytest.mark.parametrize("segs,bucket,M", [(RAGGED, 512, 3), (RAGGED, 4096, 2), (RAGGED, 96, 3), (RAGGED, 0, 3), ([5], 32, 1),
                                           ([1 << 20], 128, 4), ([33] * 1100, 64, 2)])
def test_norms_and_rule_in_one_call(G, segs, bucket, M):
    """dq_norms_choose_bits writes the norms of the separate calls and the b of dq_choose_bits, twice in a row."""
    dq = G.dq
    r = G.GpuRound(segs, bucket, M)
    ref = oracle.Layout(segs, bucket if bucket else oracle.whole_tensor_bucket(segs))
    r.set_grads(_grads(ref, segs, M, 3))
    norms = r.norms().copy()
    nbytes = dq.round_workspace_bytes(r.lay, M)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    # x half a level away from every s(b): the two fp64 sums are taken in different orders and differ by up to
    # n * 2^-53, about 1e-12 of x, so that an x on a threshold could fall on either side
    for x in (2.5, 100.5):
        rule = dq.Rule.dynamic(10, 0, 10 * float((norms.astype(np.float64) ** 2).sum()) / M / x ** 2, 1.0)
        want = r.bits(rule)
        r.g_norms.view.fill_(-1.0)
        r.set_b(1)
        dq.norms_choose_bits(r.lay, r.grads, r.stride, M, r.g_norms.view, rule, r.g_b.view, ws, nbytes, r.status)
        np.testing.assert_array_equal(r.g_norms.view.cpu().numpy().reshape(M, -1), norms)
        assert tuple(r.g_b.view.cpu().tolist()) == want
    assert r.read_status() == 0 and r.guards_intact()


@pytest.mark.parametrize("bucket", [32, 96, 160, 480, 512, 992])
def test_zero_buckets_take_no_longer_than_full_ones(G, bucket):
    """Buckets of zeros, which sparse gradients are full of, need no draws and no second reduction: a round and the
    codes alone take no longer on zeros than on normal values, for bucket lengths that are no power of two as well.
    (Best of five trains of 10 calls: 0.79 to 1.10 of the dense time; 2.7 times and more where tiles of zeros took the
    general way.)"""
    dq = G.dq
    from paper_2107_14575_b200.pipeline import Round
    M, d, b = 4, 1 << 23, 4
    rnd = Round([d], bucket, M)
    rule = dq.Rule.fixed(b)
    dense = torch.randn((M, d), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    times = {}
    for name, g in (("dense", dense), ("zeros", torch.zeros_like(dense))):
        rnd.norms_(g)
        rnd.bits_(rule)
        for call in (lambda: rnd.step_fused(g, rule, SEED, 0), lambda: rnd.norms_quantize_(g, SEED, 0)):
            best = []
            for _ in range(6):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                for _ in range(10):
                    call()
                e1.record()
                torch.cuda.synchronize()
                best.append(e0.elapsed_time(e1))
            times.setdefault(name, []).append(min(best[1:]))
    assert rnd.read_status() == 0
    for zeros, full in zip(times["zeros"], times["dense"]):
        assert zeros <= 1.25 * full, times
