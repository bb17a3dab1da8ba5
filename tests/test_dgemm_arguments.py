"""Arguments that dgemm hands to the library as they are: a transpose flag is 0
or 1 (True or False), and any other value is refused by the library's own check,
not taken as true. The operands are stand-ins of an empty product (m = 0), so
that a flag that is let through returns without touching a device."""
import types

import pytest

import paper_2609_37693_gb300 as oz

torch = pytest.importorskip("torch")


def _empty_product(rows, cols):
    return types.SimpleNamespace(dtype=torch.float64, is_cuda=True, shape=(rows, cols), device="cpu",
                                 stride=lambda i=None: (max(cols, 1), 1) if i is None else (max(cols, 1), 1)[i],
                                 numel=lambda: rows * cols, dim=lambda: 2, data_ptr=lambda: 0)


def _call(**flags):
    k, n = 8, 8
    ws = torch.empty(0, dtype=torch.uint8)
    A = _empty_product(k, 0) if flags.get("trans_a") else _empty_product(0, k)
    return oz.dgemm(A, _empty_product(n, k), oz.Plan(16, 0, k), out=_empty_product(0, n), ws=ws,
                    stream=types.SimpleNamespace(cuda_stream=0), **flags)


@pytest.mark.parametrize("flag", ["trans_a", "trans_b"])
@pytest.mark.parametrize("value", [2, -1, 7])
def test_other_flag_values_are_refused(flag, value):
    with pytest.raises(oz.OzError) as e:
        _call(**{flag: value})
    assert e.value.status == oz.OZ_ERR_INVALID_ARG


@pytest.mark.parametrize("flag", ["trans_a", "trans_b"])
def test_what_is_no_integer_is_refused(flag):
    with pytest.raises((TypeError, ValueError)):
        _call(**{flag: "yes"})


@pytest.mark.parametrize("value", [True, False, 1, 0])
def test_flags_are_taken(value):
    _call(trans_a=value, trans_b=value)
