"""Calls from host threads of their own, each with a stream and a layout, at the same time.

A thread's first CUDA call may be one of the library's: nothing else has made a context current there.
"""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [([5000], 64), ([40] * 60, 96), ([70] * 1000, 64), ([33, 64, 9000] * 200, 2048)]


@pytest.mark.parametrize("first", ["norms_", "norms_quantize_", "average_", "step", "step_fused"])
def test_fresh_threads_side_by_side(dqlib, first):
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    from paper_2107_14575_b200 import dq
    from paper_2107_14575_b200.pipeline import Round
    rule = dq.Rule.fixed(5)
    rounds = []
    for i, (segs, bucket) in enumerate(SHAPES):
        rnd = Round(segs, bucket, 2)
        g = torch.randn((2, rnd.layout.D32), generator=torch.Generator(device="cuda").manual_seed(i), device="cuda")
        rnd.norms_(g)
        rnd.bits_(rule)
        rounds.append((rnd, g, rnd.step_fused(g, rule, 1, 2).clone()))
        rnd.out.zero_()
    streams = [torch.cuda.Stream() for _ in SHAPES]
    torch.cuda.synchronize()
    gate, errors = threading.Barrier(len(SHAPES)), []

    def work(i):
        rnd, g, _ = rounds[i]
        args = {"norms_": (g,), "norms_quantize_": (g, 1, 2), "average_": (), "step": (g, rule, 1, 2),
                "step_fused": (g, rule, 1, 2)}[first]
        try:
            gate.wait()
            with torch.cuda.stream(streams[i]):
                getattr(rnd, first)(*args)
                for _ in range(100):
                    rnd.norms_quantize_(g, 1, 2)
                    rnd.average_()
        except Exception as e:                       # noqa: BLE001  (reported by the test's own thread)
            errors.append(repr(e))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(SHAPES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for rnd, _, want in rounds:
        assert rnd.read_status() == 0
        np.testing.assert_array_equal(rnd.out.cpu().numpy(), want.cpu().numpy())


def test_tables_of_different_sizes_in_bursts(dqlib):
    """The layouts' tensor tables differ in size (none, 12 KB), and with them the shared memory of the launches: no
    thread's call may narrow what another's is about to ask for.  (Bursts of calls that start together: the two have to
    meet between a thread's two runtime calls.)"""
    from paper_2107_14575_b200 import dq
    from paper_2107_14575_b200.pipeline import Round
    rounds = []
    for i, segs in enumerate([[5000], [70] * 1000, [40] * 60, [33] * 1000]):
        rnd = Round(segs, 64, 2)
        g = torch.randn((2, rnd.layout.D32), device="cuda")
        rnd.norms_(g)
        rnd.bits_(dq.Rule.fixed(5))
        rnd.norms_quantize_(g, 1, 2)
        rounds.append((rnd, g, torch.cuda.Stream()))
    torch.cuda.synchronize()
    bursts = 200
    gate, errors = threading.Barrier(len(rounds)), []

    def work(rnd, g, stream):
        with torch.cuda.stream(stream):
            for _ in range(bursts):
                gate.wait()
                try:
                    for _ in range(40):
                        rnd.norms_quantize_(g, 1, 2)
                        rnd.average_()
                except Exception as e:               # noqa: BLE001  (reported by the test's own thread)
                    errors.append(repr(e))
                stream.synchronize()
    threads = [threading.Thread(target=work, args=r) for r in rounds]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, (len(errors), errors[:3])
    assert all(rnd.read_status() == 0 for rnd, _, _ in rounds)
