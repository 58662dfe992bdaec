"""Coupling records of a path handed over as one array: the same bytes as record by record, and
every other form left to the record-by-record conversion (which accepts or refuses it)."""
import ctypes

import numpy as np
import pytest

from paper_2108_13410_gb300 import qsim as Q


@pytest.mark.parametrize("flat", [
    [(0.1, 0.2, 0.5, 0.7)], [(0.1 * k, 1 - 0.1 * k, 0.5, 0.25) for k in range(40)], [(1, 0, 1, 2)],
    [(np.float64(0.3), np.float32(0.5), 1, 0.5), (0, 0.25, 1.0, 1)], [(float("nan"), float("inf"), -0.0, 1e-320)]])
def test_same_bytes(flat):
    a = Q._path_records(flat)
    b = Q._couplings(flat, len(flat))
    assert a.tobytes() == ctypes.string_at(ctypes.addressof(b), ctypes.sizeof(b))


class _Scalar:
    """A number that converts by float() only, as a tensor on a device does."""

    def __init__(self, error):
        self.error = error

    def __float__(self):
        return 0.5

    def __array__(self, *args, **kwargs):
        raise self.error("not an array")


@pytest.mark.parametrize("error", [TypeError, RuntimeError, ValueError])
def test_numbers_numpy_refuses_are_left_alone(error):
    flat = [(_Scalar(error), 0.2, 0.5, 0.7)]
    assert Q._path_records(flat) is None
    assert Q._couplings(flat, 1)[0].g == 0.5


@pytest.mark.parametrize("flat", [
    [], [(0.1, 0.2)], [(0.1, 0.2, 0.5)], [(0.1, 0.2, 0.5, 0.7), (0.1, 0.2)], [{"g": 0.1, "lambda": 0.2}],
    [[0.1, 0.2, 0.5, 0.7]], [(0.1, 0.2, "0.5", 0.7)], [(0.1, 0.2, None, 0.7)], [(0.1, 0.2, 1j, 0.7)],
    [(True, False, True, True)], [Q.qs_couplings(1.0, 1.0, 0.1, 0.2)]])
def test_other_forms_are_left_alone(flat):
    assert Q._path_records(flat) is None
