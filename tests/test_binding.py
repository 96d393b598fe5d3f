"""What the native marshalling of binding.py accepts and refuses (no GPU: the library refuses these calls by their arguments)."""
import ctypes

import numpy as np
import pytest

from paper_2005_05758_b200 import binding

X, Y = np.zeros((2, 1, 16), np.float32), np.zeros((2, 1, 32), np.float32)


@pytest.mark.parametrize("stream", [0, ctypes.c_void_p(0), ctypes.c_void_p(None), ctypes.c_void_p(64)])
def test_streams_as_numbers_and_as_ctypes_pointers(stream):
    with pytest.raises(binding.CsbError) as e:
        binding.csb_lstm_forward([], None, X, None, None, Y, None, None, stream=stream)
    assert e.value.status == -1


def test_flags_as_a_ctypes_number():
    with pytest.raises(binding.CsbError) as e:
        binding.csb_lstm_forward([], None, X, None, None, Y, None, None, flags=ctypes.c_uint(1), stream=0)
    assert e.value.status == -1


def test_a_missing_matrix_is_the_library_s_error():
    for call in (lambda: binding.csb_lstm_forward([None], None, X, None, None, Y, None, None, stream=0),
                 lambda: binding.csb_ligru_forward([None], None, X, None, Y, None, stream=0),
                 lambda: binding.csb_lstmp_forward([None], [None], None, X, None, None, Y, None, None, stream=0)):
        with pytest.raises(binding.CsbError) as e:
            call()
        assert e.value.status == -1 and "NULL" in str(e.value)


def test_arguments_that_python_refuses():
    with pytest.raises(TypeError):
        binding.csb_lstm_forward([], None, X, None, None, Y, None, None, flags=1.5, stream=0)
    with pytest.raises(TypeError):
        binding.csb_lstm_forward([], None, X, None, None, Y, None, None, stream="0")
    with pytest.raises(IndexError):
        binding.csb_lstm_forward([None, None], [Y], X, None, None, Y, None, None, stream=0)      # a bias list that is too short
    with pytest.raises(AttributeError):
        binding.csb_lstm_forward([], None, object(), None, None, Y, None, None, stream=0)
