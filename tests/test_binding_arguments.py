"""The binding's conversion of arguments, with recorders in the place of the library's calls (no GPU)."""
import ctypes as C

import numpy as np
import pytest
import torch

_KINDS = {"p": C.c_void_p, "i": C.c_int32, "l": C.c_int64, "u": C.c_uint32, "q": C.c_uint64, "z": C.c_size_t, "f": C.c_float}
_CALLS = {
    "dq_bucket_norms": "pplippp", "dq_tensor_norms": "pplippzpp", "dq_choose_bits": "ppirppzpp",
    "dq_quantize_pack": "pplippquplpp", "dq_quantize_pack_worker": "pplippquuplpp",
    "dq_norms_quantize_pack": "pplipqupplpp", "dq_norms_quantize_pack_worker": "pplipquupplpp",
    "dq_unpack_dequant_average": "pplpipppp", "dq_unpack_average_update": "pplpipfppp",
    "dq_norms_choose_bits": "pplip" "rppzpp", "dq_quantize_average": "pplippquplpifpp",
    "dq_norms_quantize_average": "pplipqupplpifrpzpp",
}


@pytest.fixture()
def recorded(dqlib):
    """(dq, the list of the calls made): every call of a step goes to a recorder that answers DQ_OK."""
    from paper_2107_14575_b200 import dq
    dq.lib()
    made, keep, table = [], [], {}
    for name, kinds in _CALLS.items():
        types = [C.POINTER(dq.Rule) if k == "r" else _KINDS[k] for k in kinds]

        def record(*args, _name=name, _kinds=kinds):
            made.append((_name, [(a.contents.T, a.contents.b_max, a.contents.eps_hat) if k == "r" else a
                                 for a, k in zip(args, _kinds)]))
            return 0
        f = C.CFUNCTYPE(C.c_int, *types)(record)
        keep.append(f)
        table[name] = C.cast(f, C.c_void_p).value
    dq._calls.bind(table, dq.Rule)
    try:
        yield dq, made
    finally:
        dq._calls.bind({n: C.cast(getattr(dq.lib(), n), C.c_void_p).value for n in _CALLS}, dq.Rule)


@pytest.fixture()
def layout(dqlib):
    from paper_2107_14575_b200 import dq
    return dq.Layout([100], 32)


def _quantize(dq, layout, **other):
    a = dict(grads=16, worker_stride_elems=128, M=1, norms=32, dev_b=48, seed=5, step=7, packed=64,
             packed_stride_words=64, status=80, stream=0)
    a.update(other)
    dq.quantize_pack(layout, **a)


def test_integers_are_taken_by_value(recorded, layout):
    """What int() makes of an argument is its value: also of a number that lives in a tensor or an array."""
    dq, made = recorded
    for x in (3, np.int64(3), np.uint32(3), np.array(3), torch.tensor(3), torch.tensor([3]), True + 2, 3.0):
        _quantize(dq, layout, M=x, seed=x, step=x, worker_stride_elems=x, packed_stride_words=x)
        name, args = made.pop()
        assert name == "dq_quantize_pack"
        assert (args[2], args[3], args[6], args[7], args[9]) == (3, 3, 3, 3, 3), repr(x)
    _quantize(dq, layout, seed=-1, step=(1 << 40) + 9)
    _, args = made.pop()
    assert args[6] == 2 ** 64 - 1 and args[7] == 9


class _Address:
    def __init__(self, answer):
        self.answer = answer

    def data_ptr(self):
        if isinstance(self.answer, Exception):
            raise self.answer
        return self.answer


def test_an_address_is_none_an_integer_or_what_data_ptr_says(recorded, layout):
    dq, made = recorded
    t = torch.zeros(4)
    for x, want in ((None, None), (0, None), (64, 64), (t, t.data_ptr()), (_Address(128), 128), (_Address(None), None)):
        _quantize(dq, layout, grads=x, packed=x)
        _, args = made.pop()
        assert (args[1], args[8]) == (want, want), repr(x)
    for x in ("7", b"12", 3.0, np.int64(64), np.array(64), [64], _Address("64"), _Address(64.0)):
        for name in ("grads", "norms", "dev_b", "packed", "status"):
            with pytest.raises((TypeError, AttributeError)):
                _quantize(dq, layout, **{name: x})
    with pytest.raises(AttributeError, match="gone"):
        _quantize(dq, layout, grads=_Address(AttributeError("gone")))
    with pytest.raises(TypeError):
        _quantize(dq, layout, M=None)
    assert not made


def test_the_rule_is_a_rule_and_the_step_size_a_float(recorded, layout):
    dq, made = recorded
    rule = dq.Rule.dynamic(10, 3, 0.25, 0.9, 2, 9)

    class Mine(dq.Rule):
        pass
    for r in (rule, Mine(10, 3, 0.25, 0.9, 2, 9, 0)):
        dq.choose_bits(layout, 16, 1, r, 32, 48, 256, 64, stream=0)
        assert made.pop()[1][3] == (10, 9, 0.25)
    for r in (bytes(rule), bytearray(bytes(rule)), np.zeros(5), None, 4):
        with pytest.raises((TypeError, C.ArgumentError)):
            dq.choose_bits(layout, 16, 1, r, 32, 48, 256, 64, stream=0)
    for lr in (0.5, np.float32(0.5), torch.tensor(0.5), "0.5"):
        dq.unpack_average_update(layout, 16, 4, 32, 1, 48, lr, 64, 80, stream=0)
        assert made.pop()[1][6] == 0.5
    for lr in (None, "x"):
        with pytest.raises((TypeError, ValueError)):
            dq.unpack_average_update(layout, 16, 4, 32, 1, 48, lr, 64, 80, stream=0)
    assert not made
