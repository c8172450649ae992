"""pes_auto_arith and the arithmetic by name, without a GPU: argument checks and the kinds of
polynomial the automatic arithmetic tells apart."""
import ctypes
import itertools

import numpy as np
import pytest

from paper_2101_10881_gb300 import pes, synth


@pytest.fixture(scope="module", autouse=True)
def built():
    pes.build()


def test_wide_and_narrow_polynomials():
    assert pes.auto_arith(synth.supports_p2(), 152, 10) == "tensor"
    assert pes.auto_arith(synth.supports_p3(128), 152, 4) == "tensor"
    assert pes.auto_arith(synth.supports_p3(128), 152, 2) == "int"
    assert pes.auto_arith([list(range(64))], 152, 10) == "int"
    assert pes.auto_arith([], 152, 10) == "int"


# degree and products of two variables on either side of the line, or no line at all
LINES = [(10, 100, 254), (10, 300, 47), (10, 600, 18), (8, 100, 356), (8, 300, 88), (8, 700, 38), (4, 150, 298),
         (4, 300, 130), (4, 400, 183), (4, 1100, 6), (5, 256, 118), (5, 275, 166)]
NEVER = [(10, 55), (8, 71), (8, 520), (4, 135), (4, 700), (5, 255), (5, 300), (5, 900), (3, 152), (2, 152), (1, 152)]


@pytest.mark.parametrize("k,d,N", LINES)
def test_lines(k, d, N):
    assert pes.auto_arith([[0, 1]] * (N - 1), d, k) == "int"
    assert pes.auto_arith([[0, 1]] * N, d, k) == "tensor"


@pytest.mark.parametrize("k,d", NEVER)
def test_degrees_that_stay_on_the_integer_pipe(k, d):
    assert pes.auto_arith([[0, 1]] * 50000, d, k) == "int"


def test_arguments_checked_on_host():
    L = pes.lib()
    ptr = np.array([0, 2, 2], dtype=np.int32)
    a = ctypes.c_int32()
    assert L.pes_auto_arith(pes._ip32(ptr), 2, 10, 10, ctypes.byref(a)) == 1  # an empty monomial
    assert L.pes_auto_arith(pes._ip32(ptr), 1, -1, 10, ctypes.byref(a)) == 1
    assert L.pes_auto_arith(None, 1, 10, 10, ctypes.byref(a)) == 1
    assert L.pes_auto_arith(pes._ip32(ptr), 1, 10, 6, ctypes.byref(a)) == 2
    assert L.pes_get_plan_arith(None, ctypes.byref(a)) == 1
    for k in (1, 2, 3):
        with pytest.raises(pes.PesError) as e:
            pes.Plan([[0, 1]], 2, 8, k, arith="tensor")
        assert e.value.code == 1
    with pytest.raises(pes.PesError) as e:
        pes.Plan([[0, 1]], 2, 8, 10, arith=3)
    assert e.value.code == 1


def test_same_digits_are_rounded_for_either_integer_form():
    rng = np.random.default_rng(2)
    k, n, d = 4, 2, 3
    L = (53 * k + 28 + 27) // 28 + 1
    grids = rng.integers(-3, 3, size=(n + 1, d + 1))
    acc = rng.integers(-2 ** 40, 2 ** 40, size=(n + 1, d + 1, L))
    a, b = (pes.round_sums_host(k, n, d, grids, acc, arith=name) for name in ("int", "tensor"))
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
