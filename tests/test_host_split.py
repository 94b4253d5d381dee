"""Host-only check of the split of a 2 x 2 factor into phases and a real rotation
(the decision that sends a one-qubit operator to the rotation passes): unitary
and rank-one factors reproduce to 1e-10, and a factor with an entry that is not
finite is never taken, wherever the entry stands."""
import ctypes

import numpy as np
import pytest

import workloads as W

SYMBOL = "_ZN3qsa14split_rotationERKSt5arrayISt7complexIdELm4EEPdS6_PS2_S7_"


@pytest.fixture(scope="module")
def split():
    import __graft_entry__
    f = getattr(ctypes.CDLL(__graft_entry__._build_module().build()), SYMBOL)
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_void_p] * 5

    def call(F):
        F = np.ascontiguousarray(F, dtype=np.complex128)
        c, s, p, q = np.zeros(1), np.zeros(1), np.zeros(2, dtype=np.complex128), np.zeros(2, dtype=np.complex128)
        ok = f(*(a.ctypes.data for a in (F, c, s, p, q)))
        return ok, ok and np.diag(p) @ np.array([[c[0], -s[0]], [s[0], c[0]]]) @ np.diag(q)
    return call


FACTORS = [W.haar_unitary(2, np.random.default_rng(1)), np.eye(2), W.X, W.H, np.diag([1, 1j]),
           np.array([[0.6, 0.8], [0, 0]])]


@pytest.mark.parametrize("f", range(len(FACTORS)))
def test_split_reproduces(split, f):
    ok, got = split(FACTORS[f])
    assert ok and np.abs(got - FACTORS[f]).max() <= 1e-10


@pytest.mark.parametrize("f", range(len(FACTORS)))
@pytest.mark.parametrize("bad", [np.nan, complex(0, np.nan), np.inf])
def test_split_refuses_what_is_not_finite(split, f, bad):
    for i in range(4):
        F = np.array(FACTORS[f], dtype=np.complex128)
        F.flat[i] = bad
        assert not split(F)[0], (i, F)
