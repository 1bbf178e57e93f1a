"""Where a curve runs the column form of the s-contraction, as the library reports it."""
import ctypes

import pytest

from paper_2301_11704_gb300 import _native
from tests.test_capi_cpu import _params


@pytest.mark.parametrize("kw,length", [
    (dict(precision=1, ns=63), 0), (dict(precision=1, ns=64), 128), (dict(precision=1, ns=129), 256),
    (dict(precision=1, ns=16384), 16384), (dict(precision=1, ns=16385), 0), (dict(precision=2, nx=64, ns=1024), 1024),
    (dict(precision=0, ns=64), 128), (dict(precision=0, ns=8192), 8192), (dict(precision=0, ns=8193), 0),
    (dict(precision=0, ns=600, symmetry=5), 1024), (dict(precision=0, ns=600, scheme=1), 1024),
    (dict(precision=1, ns=1024, s_transform=1), 0), (dict(precision=1, ns=1024, s_transform=5), 0),
    (dict(precision=1, ns=300, launch=1), 0), (dict(nx=24), -1),
])
def test_column_length(kw, length):
    assert _native.load().ks_curve_column_length(ctypes.byref(_params(**kw))) == length
