"""Rounds in which a warp takes its tiles through the workers, against the separate calls, bit for bit.

Layouts with few tiles go to another kernel, so these have the small tensors of every edge and one of 3.3 million
elements; every test asserts the route that it means.  The separate calls are held against the oracle elsewhere.
"""
import numpy as np
import pytest
import torch

import oracle
import route_util

pytestmark = pytest.mark.gpu

SEED = 0x3A_2B0_17D5
RAGGED = [70, 1, 1023, 1024, 1025, 0, 4097, 31, 2048, 3 * 4096 + 77, 32, 9000]
BIG = RAGGED + [3300000]
MANY = [33] * 1100 + [3300000]                     # the tensor table does not fit the shared memory
LIMIT_NS = 50_000_000


@pytest.fixture(scope="module")
def G(dqlib):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    import gpu_util
    return gpu_util


@pytest.fixture(scope="module")
def by_warps(tmp_path_factory):
    route = route_util.compile_route(tmp_path_factory.mktemp("route"))
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def check(r, bucket, lost=False, given=None):
        """given: the layout's buckets, but for a call whose norms are given."""
        groups = r.lay.D32 // 32
        b = 0 if given else bucket
        assert route(groups, r.lay.nb, b, r.M, sms, lost, r.linf) == route_util.WARPS
    return check


def _round(G, segs, bucket, M, b, linf=False, seed=0):
    """Normal values of very different scales, a tensor of zeros, a bucket of tiny entries, NaN in the padding."""
    r = G.GpuRound(segs, bucket, M, norm=G.dq.NORM_LINF if linf else G.dq.NORM_L2)
    gen = torch.Generator(device="cuda").manual_seed(100 * M + b + seed)
    g = torch.full((M, r.stride), float("nan"), device="cuda")
    at = 0
    r.offsets, r.linf = [], linf
    for i, n in enumerate(segs):
        r.offsets.append(at)
        g[:, at: at + n] = torch.randn((M, n), generator=gen, device="cuda") * 10.0 ** (i % 5 - 2)
        at += -(-n // 32) * 32
    if len(segs) > 8:
        g[:, r.offsets[8]: r.offsets[8] + segs[8]] = 0.0
        g[0, r.offsets[4]: r.offsets[4] + segs[4]] *= 1e-30
    r.grads = g
    r.set_b(b)
    r.ws_bytes = G.dq.round_workspace_bytes(r.lay, M)
    r.ws = torch.zeros(r.ws_bytes, dtype=torch.uint8, device="cuda")
    return r


def _one_call(G, r, whole, lr=None, rule=None):
    if whole:
        G.dq.norms_quantize_average(r.lay, r.grads, r.stride, r.M, r.g_b.view, SEED, 9, r.g_norms.view, r.g_packed.view, r.pstride,
                                    r.g_out.view, rule or G.dq.Rule.fixed(7), r.ws, r.ws_bytes, r.status, lr=lr)
    else:
        G.dq.quantize_average(r.lay, r.grads, r.stride, r.M, r.g_norms.view, r.g_b.view, SEED, 9, r.g_packed.view, r.pstride,
                              r.g_out.view, r.status, lr=lr)


def _equals_the_separate_calls(G, r, b, status=0):
    r.set_b(b)
    norms = r.norms().copy()
    packed = r.quantize(SEED, 9, fill=-1).copy()
    avg = r.average(fill=1.0).copy()
    x0 = np.linspace(-1, 1, r.lay.D32, dtype=np.float32)
    upd = r.update(0.125, x0).copy()
    for whole in (False, True):
        for lr, want in ((None, avg), (0.125, upd)):
            r.set_b(b)
            r.g_packed.view.fill_(-1)
            if whole:
                r.g_norms.view.fill_(-1.0)
            r.g_out.view.copy_(torch.from_numpy(x0))
            _one_call(G, r, whole, lr)
            np.testing.assert_array_equal(r.g_norms.view.cpu().numpy().reshape(r.M, -1), norms)
            np.testing.assert_array_equal(r.g_packed.view.cpu().numpy().view(np.uint32).reshape(r.M, -1), packed)
            np.testing.assert_array_equal(r.g_out.view.cpu().numpy(), want)
    assert r.read_status() == status and r.guards_intact()
    return norms, avg


WIDTHS = [(BIG, bucket, b, linf) for bucket, linf in ((256, False), (512, True), (2048, False)) for b in range(1, 17)]
WIDTHS += [(BIG, 0, b, False) for b in (1, 2, 5, 9, 11, 16)] + [(BIG, 1056, b, False) for b in (3, 7)]
WIDTHS += [(BIG, bucket, b, linf) for bucket, linf in ((96, False), (480, False), (992, True), (4096, False)) for b in (1, 3, 6, 9, 14)]
WIDTHS += [(MANY, bucket, b, False) for bucket, b in ((64, 7), (2048, 5), (480, 4), (0, 6))]


@pytest.mark.parametrize("segs,bucket,b,linf", WIDTHS)
def test_equals_the_separate_calls(G, by_warps, segs, bucket, b, linf):
    r = _round(G, segs, bucket, 3, b, linf)
    by_warps(r, bucket)
    by_warps(r, bucket, given=True)
    _equals_the_separate_calls(G, r, b)


@pytest.mark.parametrize("bucket", [512, 96, 480, 2048, 4096, 0, 1056])
def test_lost_first_wait_and_a_call_that_cannot_run(G, by_warps, bucket):
    """A lost wait raises DQ_STAT_WAIT and nothing else; a b outside 1..16 or a stream too short for b write no output
    but still get their successor; the next call is right."""
    dq = G.dq
    b = 4
    r = _round(G, BIG, bucket, 3, b)
    r.grads = torch.nan_to_num(r.grads)
    for given in (False, True):
        by_warps(r, bucket, given=given)
        by_warps(r, bucket, lost=True, given=given)
    norms, _ = _equals_the_separate_calls(G, r, b)
    short = r.pstride // 16 * 8                     # words of half the widest codes
    for whole in (False, True):
        r.set_b(b)
        r.clear_status()
        dq.debug_set_wait_limits(LIMIT_NS, True)
        try:
            _one_call(G, r, whole, rule=dq.Rule.fixed(6))
            torch.cuda.synchronize()
        finally:
            dq.debug_set_wait_limits()
        assert r.read_status() == dq.STAT_WAIT and r.guards_intact()
        for bad, why in ((17, dq.STAT_BAD_BITS), (0, dq.STAT_BAD_BITS), (9, dq.STAT_CAPACITY)):
            full = r.pstride
            r.pstride = short if why == dq.STAT_CAPACITY else full
            r.g_packed.view.fill_(-7)
            r.g_out.view.fill_(3.0)
            r.set_norms(norms)
            r.set_b(bad)
            r.clear_status()
            _one_call(G, r, whole, rule=dq.Rule.fixed(6))
            r.pstride = full
            assert r.read_status() == why and r.guards_intact()
            assert bool((r.g_packed.view == -7).all()) and bool((r.g_out.view == 3.0).all())
            assert not whole or r.g_b.view.tolist() == [6, 31]
        r.clear_status()
        _equals_the_separate_calls(G, r, b)


@pytest.mark.parametrize("b", [1, 2, 4, 5, 8, 11])
@pytest.mark.parametrize("bucket,linf", [(32, False), (96, False), (512, False), (512, True), (2048, False), (4096, False), (1056, False), (0, False)])
def test_buckets_that_are_not_finite(G, by_warps, bucket, linf, b):
    """Their averages are NaN and their neighbours' are not; norms found by the call and given alike."""
    M = 3
    r = _round(G, BIG, bucket, M, b, linf)
    by_warps(r, bucket)
    by_warps(r, bucket, given=True)
    ref = oracle.Layout(BIG, bucket if bucket else oracle.whole_tensor_bucket(BIG))
    r.grads = torch.nan_to_num(r.grads)
    hit = [k for k in range(ref.nb) if k % 7 == 1][:400] + [ref.nb - 1]
    dirty = np.zeros(ref.D32, bool)
    for i, k in enumerate(hit):
        at, n = int(ref.bucket_start[k]), int(ref.bucket_len[k])
        r.grads[i % M, at + (13 * i) % n] = (float("nan"), float("inf"), float("-inf"))[i // M % 3]
        dirty[at: at + n] = b > 1
    norms, avg = _equals_the_separate_calls(G, r, b, status=G.dq.STAT_NONFINITE)
    assert set(np.flatnonzero(~np.isfinite(norms).all(axis=0)).tolist()) == set(hit)
    np.testing.assert_array_equal(np.isnan(avg), dirty)


@pytest.mark.parametrize("bucket,b", [(64, 2), (64, 3), (64, 4), (64, 5), (64, 8), (64, 12), (64, 16), (512, 4), (2048, 6), (96, 3)])
def test_averages_up_to_the_top_of_the_range(G, by_warps, bucket, b):
    """Entries of 2^-90 to 2^120 in neighbouring buckets: finite, and the one of the average from the words."""
    r = _round(G, BIG, bucket, 3, b)
    by_warps(r, bucket)
    expo = torch.tensor([0, 90, 104, 108, 111, 116, 120, -90], device="cuda")
    of = expo[torch.arange(r.lay.D32, device="cuda") // bucket % 8]
    gen = torch.Generator(device="cuda").manual_seed(b)
    r.grads = torch.ldexp(torch.rand((3, r.lay.D32), generator=gen, device="cuda") * 2 - 1, of)
    _, avg = _equals_the_separate_calls(G, r, b)
    assert np.isfinite(avg).all()


@pytest.mark.parametrize("bucket,b", [(480, 4), (512, 4), (2048, 5), (4096, 6), (512, 7), (0, 4)])
def test_repeated_passes_write_the_same_bits(G, by_warps, bucket, b):
    """A stage is refilled while its warp may still be reading it unless the two are ordered: passes over two sets of
    gradients in turn, without a pause, give the same words and averages every time."""
    M, sets = 8, []
    for i in range(2):
        r = _round(G, [6_300_001, 50001], bucket, M, b, seed=i)
        r.grads = torch.nan_to_num(r.grads)
        by_warps(r, bucket)
        by_warps(r, bucket, given=True)
        r.norms()
        r.quantize(SEED, 9, fill=-1)
        r.average()
        sets.append((r, r.g_packed.view.clone(), r.g_out.view.clone(), r.g_norms.view.clone()))
    for k in range(16):
        for r, *_ in sets:
            _one_call(G, r, k % 2 == 0, rule=G.dq.Rule.fixed(b))
        for r, packed, out, norms in sets:
            assert torch.equal(r.g_packed.view, packed) and torch.equal(r.g_out.view, out) and torch.equal(r.g_norms.view, norms)
    assert all(r.read_status() == 0 and r.guards_intact() for r, *_ in sets)
