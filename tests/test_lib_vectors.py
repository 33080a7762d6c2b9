"""The four-vectors that the binding hands to the library: any sequence of numbers, converted when
the call is made."""
import numpy as np
import torch

from paper_2505_14399_gb300 import _lib as L


def test_sequences_of_any_number_type():
    for v in ((4, 6, 2, 8), [4, 6, 2, 8], np.array([4, 6, 2, 8]), torch.tensor([4, 6, 2, 8]),
              [np.array(4), np.array(6), 2.0, np.int8(8)]):
        assert list(L.ivec(v)) == [4, 6, 2, 8]
        assert list(L.dvec(v)) == [4.0, 6.0, 2.0, 8.0]


def test_values_are_read_at_every_call():
    v = [torch.tensor(float(i)) for i in range(4)]
    assert list(L.dvec(v)) == [0.0, 1.0, 2.0, 3.0] and list(L.ivec(v)) == [0, 1, 2, 3]
    v[0].fill_(7.0)
    assert list(L.dvec(v))[0] == 7.0 and list(L.ivec(v))[0] == 7
    w = [np.zeros(()) for _ in range(4)]
    assert list(L.dvec(w)) == [0.0] * 4
    w[3][...] = 5.0
    assert list(L.dvec(w))[3] == 5.0


def test_signs_of_zero_are_kept():
    assert np.signbit(np.array(list(L.dvec((0.0, -0.0, 0.0, -0.0))))).tolist() == [0, 1, 0, 1]
    assert np.signbit(np.array(list(L.dvec((-0.0, 0.0, -0.0, 0.0))))).tolist() == [1, 0, 1, 0]
