"""Sizes that fock_shellpairs_build cannot number are refused before any work
(on any machine: no CUDA call is made)."""
import ctypes

import numpy as np

import molgen
from paper_2407_21445_gb300 import fock as fb


def test_more_coefficients_than_an_int_counts():
    """f shells of eight primitives whose canonical pairs hold more than 2^31
    Hermite coefficients."""
    per_pair = 64 * fb.fock_hermite_count(3, 3)
    ns = int(np.sqrt(2 * 2.0 ** 31 / per_pair)) + 2
    assert per_pair * ns * (ns + 1) // 2 > 2 ** 31
    bas = molgen.single_shell_basis([(3, np.zeros(3), 0.1 * 2.0 ** np.arange(8), np.ones(8)) for _ in range(ns)])
    arr = fb._BasisArrays(bas)
    out = ctypes.c_void_p(1)
    rc = fb.lib().fock_shellpairs_build(ctypes.byref(arr.desc), None, 1e-10, None, ctypes.byref(out))
    assert rc == 1 and out.value is None  # FOCK_ERR_INVALID_ARG
