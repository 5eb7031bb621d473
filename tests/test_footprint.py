"""Device bytes an element takes in FP64.

A problem that fits a device memory (or a server's budget) with the metrics and the
inverse mass alone, from which a stage forms what it needs, fits with the operators
that the kernels store per element too.
"""

import ctypes

import pytest

from paper_2005_02516_gb300 import esdg
from test_library_cpu import _cfg, _lib

# (method, N, rule, mass, forcing): bytes an element without such stored operators
# (16-point rules and below: with the pair operator and the inverse's products)
BYTES = {
    ("modal", 1, "symmetric", "exact", "none"): 5396,
    ("modal", 1, "symmetric", "exact", "mms_sine"): 5956,
    ("modal", 1, "symmetric", "weight_adjusted", "none"): 3284,
    ("modal", 1, "symmetric", "weight_adjusted", "mms_sine"): 3332,
    ("modal", 1, "collapsed", "exact", "none"): 5780,
    ("modal", 1, "collapsed", "exact", "mms_sine"): 6356,
    ("modal", 1, "collapsed", "weight_adjusted", "none"): 3412,
    ("modal", 1, "collapsed", "weight_adjusted", "mms_sine"): 3476,
    ("modal", 2, "symmetric", "exact", "none"): 9508,
    ("modal", 2, "symmetric", "exact", "mms_sine"): 10372,
    ("modal", 2, "symmetric", "weight_adjusted", "none"): 5732,
    ("modal", 2, "symmetric", "weight_adjusted", "mms_sine"): 5828,
    ("modal", 2, "collapsed", "exact", "none"): 10916,
    ("modal", 2, "collapsed", "exact", "mms_sine"): 12340,
    ("modal", 2, "collapsed", "weight_adjusted", "none"): 6116,
    ("modal", 2, "collapsed", "weight_adjusted", "mms_sine"): 6260,
    ("modal", 3, "symmetric", "exact", "none"): 14716,
    ("modal", 3, "symmetric", "exact", "mms_sine"): 16444,
    ("modal", 3, "symmetric", "weight_adjusted", "none"): 8124,
    ("modal", 3, "symmetric", "weight_adjusted", "mms_sine"): 8316,
    ("modal", 3, "collapsed", "exact", "none"): 18300,
    ("modal", 3, "collapsed", "exact", "mms_sine"): 20604,
    ("modal", 3, "collapsed", "weight_adjusted", "none"): 10172,
    ("modal", 3, "collapsed", "weight_adjusted", "mms_sine"): 10428,
    ("modal", 4, "symmetric", "exact", "none"): 19996,
    ("modal", 4, "symmetric", "exact", "mms_sine"): 22300,
    ("modal", 4, "symmetric", "weight_adjusted", "none"): 10844,
    ("modal", 4, "symmetric", "weight_adjusted", "mms_sine"): 11100,
    ("modal", 4, "collapsed", "exact", "none"): 6812,
    ("modal", 4, "collapsed", "exact", "mms_sine"): 7212,
    ("modal", 4, "collapsed", "weight_adjusted", "none"): 5852,
    ("modal", 4, "collapsed", "weight_adjusted", "mms_sine"): 6252,
    ("modal", 5, "symmetric", "exact", "none"): 8452,
    ("modal", 5, "symmetric", "exact", "mms_sine"): 8852,
    ("modal", 5, "symmetric", "weight_adjusted", "none"): 6596,
    ("modal", 5, "symmetric", "weight_adjusted", "mms_sine"): 6996,
    ("modal", 5, "collapsed", "exact", "none"): 9860,
    ("modal", 5, "collapsed", "exact", "mms_sine"): 10436,
    ("modal", 5, "collapsed", "weight_adjusted", "none"): 8004,
    ("modal", 5, "collapsed", "weight_adjusted", "mms_sine"): 8580,
    ("sbp", 1, "symmetric", "exact", "none"): 2284,
    ("sbp", 1, "symmetric", "exact", "mms_sine"): 2380,
    ("sbp", 2, "symmetric", "exact", "none"): 4140,
    ("sbp", 2, "symmetric", "exact", "mms_sine"): 4300,
    ("sbp", 3, "symmetric", "exact", "none"): 9388,
    ("sbp", 3, "symmetric", "exact", "mms_sine"): 9676,
    ("sbp", 4, "symmetric", "exact", "none"): 12780,
    ("sbp", 4, "symmetric", "exact", "mms_sine"): 13132,
    ("sbp", 5, "symmetric", "exact", "none"): 26028,
    ("sbp", 5, "symmetric", "exact", "mms_sine"): 26572,
}
POINTS_25 = [k for k in BYTES if k[0] == "modal" and k[1:3] in ((4, "collapsed"), (5, "symmetric"))]


def _context(method, N, rule, mass, forcing, nx, ny=32):
    c = _cfg(N=N, nx=nx, ny=ny, warp=0.05,
             rule=esdg.ESDG_RULE_SYMMETRIC if rule == "symmetric" else esdg.ESDG_RULE_COLLAPSED,
             mass=esdg.ESDG_MASS_EXACT if mass == "exact" else esdg.ESDG_MASS_WEIGHT_ADJUSTED,
             method=esdg.ESDG_METHOD_SBP if method == "sbp" else esdg.ESDG_METHOD_MODAL)
    if forcing != "none":
        c.forcing = esdg.ESDG_FORCING_MMS_SINE
        c.mms_amp = c.mms_bamp = 0.1
    h = ctypes.c_void_p()
    lib = _lib()
    assert lib.esdg_build_operators(ctypes.byref(c), ctypes.byref(h)) == 0
    return lib, h


def _bytes(lib, h):
    K, nb = ctypes.c_int(), ctypes.c_size_t()
    assert lib.esdg_sizes(h, ctypes.byref(K), None, None, None, ctypes.byref(nb)) == 0
    return K.value, nb.value


def _per_element(key, change=lambda lib, h: None):
    sizes = []
    for nx in (16, 32):
        lib, h = _context(*key, nx)
        change(lib, h)
        sizes.append(_bytes(lib, h))
        lib.esdg_destroy(h)
    (k0, b0), (k1, b1) = sizes
    return (b1 - b0) / (k1 - k0)


@pytest.mark.parametrize("key", [k for k in BYTES if k not in POINTS_25], ids=str)
def test_an_element_takes_no_more_than_without_stored_operators(key):
    # (4 bytes: DG-SBP keeps one word of scales)
    assert _per_element(key) <= BYTES[key] + 4


def _compact(lib, h):
    assert lib.esdg_prefer_compact(h) == 0


@pytest.mark.parametrize("key", POINTS_25, ids=str)
def test_the_compact_form_takes_no_more_than_without_stored_operators(key):
    assert _per_element(key, _compact) <= BYTES[key]
    assert _per_element(key) > BYTES[key]  # the stored form is the one of small problems


@pytest.mark.parametrize("key", [k for k in BYTES if k not in POINTS_25][::7], ids=str)
def test_other_rules_have_one_form(key):
    assert _per_element(key, _compact) == _per_element(key)


def test_a_large_problem_takes_the_compact_form():
    # 24.6 KB an element with the stored operators: 16 GiB are reached at 700 thousand
    key = ("modal", 4, "collapsed", "exact", "none")
    lib, h = _context(*key, 720, 490)
    K, nb = _bytes(lib, h)
    lib.esdg_destroy(h)
    assert K == 705600 and nb <= K * BYTES[key]
