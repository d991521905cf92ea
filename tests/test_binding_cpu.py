"""The native half of the binding checks its arguments before it calls the library (no GPU needed)."""
import pytest
import torch

from paper_2607_23815_b200 import kvattn


class _NoPool:
    ptr = None


def test_tensors_must_be_contiguous_and_on_the_gpu():
    t, i = torch.zeros(2, 4, 64, dtype=torch.bfloat16), torch.zeros(2, 8, dtype=torch.int32)
    dec = lambda q: kvattn.attn_decode(_NoPool, q, i, i[0], 5, 1.0, t, t, None, 0)
    with pytest.raises(AssertionError, match="CUDA"):
        dec(t)
    with pytest.raises(AssertionError, match="contiguous"):
        dec(t.transpose(0, 1))
    with pytest.raises(TypeError, match="torch tensor"):
        dec([1, 2])


def test_errors_of_the_library_come_back_as_kverror():
    with pytest.raises(kvattn.KvError) as e:                              # no pool: refused by the library itself
        kvattn.attn_mixed(_NoPool, 8, 1.0, None, None, None, 0)
    assert e.value.status == kvattn.KV_ERR_INVALID
    with pytest.raises(TypeError):                                        # a structure of another kind
        kvattn.attn_mixed(_NoPool, 8, 1.0, kvattn.DecodeArgs(), None, None, 0)
