"""What PagedAttention's calls with tensors refuse before they reach the device, against the calls through addresses."""
import numpy as np
import pytest
import torch

import paper_2507_17769_b200 as ps
from paper_2507_17769_b200 import session


def host_session():
    """A PagedAttention without a pool: what its calls do up to the library, which refuses a null pool before any device call."""
    pa = object.__new__(ps.PagedAttention)
    pa.torch, pa._calls = torch, ps.binding.calls()
    pa._tensor_calls, pa._tensor = session.torch_calls(), torch.Tensor
    pa.device, pa.shape = torch.device("cpu"), ps.binding.make_shape(8, 2, 64)
    pa.pool, pa.kv, pa._plan = torch.empty(16, dtype=torch.uint8), 0, None
    pa._stream = lambda: 0
    return pa


class Sub(torch.Tensor):  # (these take the calls through addresses)
    pass


@pytest.mark.parametrize("length", [2.5, np.float64(2), True, "3", None, torch.tensor(2.5)], ids=repr)
def test_gather_takes_no_length_that_is_not_an_integer(length):
    row = torch.zeros(4, dtype=torch.int32)
    for table in (row, row.as_subclass(Sub)):
        with pytest.raises(TypeError):
            host_session().gather(table, length)


def test_lengths_of_integer_types_are_taken():
    row = torch.zeros(4, dtype=torch.int32)
    for length in (3, np.int64(3), np.int32(3), torch.tensor(3)):
        for table in (row, row.as_subclass(Sub)):
            with pytest.raises(ps.PsError) as e:  # (as far as the null pool)
                host_session().gather(table, length)
            assert e.value.status == ps.binding.PS_ERR_INVALID


def test_a_closed_pool_is_reported_as_the_library_does():
    pa = host_session()
    pa.kv = None
    k, row = torch.zeros((1, 2, 64), dtype=torch.bfloat16), torch.zeros((1, 4), dtype=torch.int32)
    for cast in (lambda x: x, lambda x: x.as_subclass(Sub)):
        for call in (lambda: pa.write(cast(k), cast(k), cast(row), [0], [1]), lambda: pa.gather(cast(row), 1)):
            with pytest.raises(ps.PsError) as e:
                call()
            assert e.value.status == ps.binding.PS_ERR_INVALID
