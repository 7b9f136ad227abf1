"""Forms of arguments that ctypes takes beside plain numbers, and tensor subclasses
with a say of their own: the C++ marshalling takes them too, without a GPU."""
import ctypes

import pytest
import torch

from test_bind import _scan, rs  # noqa: F401  (the fixture that builds the library)


class _As:
    def __init__(self, x):
        self._as_parameter_ = x


def test_ctypes_numbers(rs):  # noqa: F811
    for B in (ctypes.c_int(0), _As(0), _As(ctypes.c_int(0)), _As(_As(0))):
        _scan(rs, B=B)
    with pytest.raises(rs.RespecError, match="negative B"):
        _scan(rs, B=ctypes.c_int(-1))
    with pytest.raises(rs.RespecError, match="scale"):
        rs.rs_tree_verify_attn(16, 16, 16, ctypes.c_int64(0), 16, 16, 16, 16, _As(1), 0, 4, 4, 64, ctypes.c_float(-1.0), 16, 16, 16,
                               None, stream=0)
    with pytest.raises(rs.RespecError, match="scale"):
        rs.rs_tree_verify_attn(16, 16, 16, 0, 16, 16, 16, 16, 1, 0, 4, 4, 64, _As(-1.0), 16, 16, 16, None, stream=0)
    for bad in (ctypes.c_int64(0), ctypes.c_float(0), _As("x"), _As(None)):
        with pytest.raises(ctypes.ArgumentError):
            _scan(rs, B=bad)


def test_parameters_behind_as_parameter(rs):  # noqa: F811
    _scan(rs, p=_As(rs.params()))
    with pytest.raises(rs.RespecError, match="top_c=9"):
        _scan(rs, p=_As(rs.params(top_c=9)))

    class More(rs.rs_params):
        pass

    _scan(rs, p=More.from_buffer_copy(rs.params()))


def test_stream_handles(rs):  # noqa: F811
    class Stream:
        def __init__(self, h):
            self.cuda_stream = h

    loop = _As(None)
    loop._as_parameter_ = loop
    with pytest.raises(ctypes.ArgumentError):
        _scan(rs, stream=Stream(loop))
    for h in (0, 4096, None, ctypes.c_void_p(4096), ctypes.c_void_p(None), _As(4096)):
        _scan(rs, stream=Stream(h))
    with pytest.raises(ctypes.ArgumentError):
        _scan(rs, stream=Stream(1.5))


def test_addresses_that_are_not_plain_numbers(rs):  # noqa: F811
    class Like:
        is_cuda, device = True, "like"

        def __init__(self, address):
            self.address = address

        def is_contiguous(self):
            return True

        def data_ptr(self):
            return self.address

    for a in (4096, None, ctypes.c_void_p(4096), ctypes.c_void_p(None)):
        _scan(rs, tokens=Like(a))
    with pytest.raises(rs.RespecError, match="null pointer"):   # None is the null address, not one that is there
        _scan(rs, tokens=Like(None), B=1)
    with pytest.raises(rs.RespecError, match="null pointer"):
        _scan(rs, tokens=Like(ctypes.c_void_p(None)), B=1)
    with pytest.raises(ctypes.ArgumentError):
        _scan(rs, tokens=Like(1.5))


def test_subclasses_answer_for_themselves(rs):  # noqa: F811
    class Sub(torch.Tensor):
        is_cuda = True

        def is_contiguous(self):
            return True

        def data_ptr(self):
            return 4096

    _scan(rs, tokens=torch.zeros(4, dtype=torch.int32).as_subclass(Sub))
    with pytest.raises(ValueError, match="CUDA"):  # a Parameter is a plain tensor
        _scan(rs, tokens=torch.nn.Parameter(torch.zeros(4)))


def test_an_index_of_no_tokens_still_needs_its_offsets(rs):  # noqa: F811
    # the build reads them on the device whatever the total
    class Index:
        is_cuda, device = True, "like"

        def is_contiguous(self):
            return True

        def data_ptr(self):
            return 4096

        def numel(self):
            return 1 << 30

        def element_size(self):
            return 1

    with pytest.raises(rs.RespecError, match="null pointer") as e:
        rs.rs_match_index_build(None, None, 1, 4, 0, Index(), stream=0)
    assert e.value.status == rs.RS_ERR_INVALID_ARG
    rs.rs_match_index_build(None, None, 0, 4, 0, Index(), stream=0)
