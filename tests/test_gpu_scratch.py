"""Temporaries of the operators and of the tuner when an allocation fails while
the library's pool holds memory: the pool is given back and the call goes on.
The failure is made on the host (dw_test_refuse)."""
import os
import subprocess
import sys

import pytest

from helpers import ROOT

pytestmark = pytest.mark.gpu

CHILD = r'''
import ctypes, os, sys
import numpy as np
sys.path.insert(0, os.environ["REPO"])
import torch
from paper_2001_05218_gb300 import dw, inputs as I
SCRATCH = 3  # as in csrc/dw_internal.h
refuse = ctypes.CDLL(dw.LIB_PATH).dw_test_refuse
dims = (6, 10, 6, 6)
U, psi = I.gauge_field(dims, "exp", 81, 1, 0.4), I.gaussian_spinor(dims, 81, 2)
Ug = dw.gauge(dims, 0.12, U)
x, y, z = dw.spinor(dims, psi), dw.spinor(dims), dw.spinor(dims)
dw.apply(Ug, x, y, normal=True)
assert refuse(SCRATCH, 1) == dw.DW_OK
dw.apply(Ug, x, z, normal=True)  # one temporary
assert np.array_equal(y.download(), z.download())
assert refuse(SCRATCH, 1) == dw.DW_OK
s, st = dw.cg_solve(Ug, x, z, dw.params(tol=1e-10, inner="f64"))  # the tuner's fields
assert s == dw.DW_OK
'''


def test_pool_is_given_back_when_an_allocation_fails(tmp_path):
    env = dict(os.environ, DW_TUNE_CACHE=str(tmp_path / "tune.txt"), REPO=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    assert "f64c18/r1/6x10x6x6" in (tmp_path / "tune.txt").read_text()  # tuned all the same
