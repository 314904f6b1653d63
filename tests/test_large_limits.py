"""Sizes hpeel_mphf_build_large refuses before it touches the device (no GPU
needed): ids at or past the width of a vertex record's id sum."""
import ctypes

import pytest

from paper_1312_0526_gb300 import build as hpbuild

import paper_1312_0526_gb300 as hp


@pytest.fixture(scope="module")
def lib():
    hpbuild.build()
    return hp.lib()


def _call(lib, n, gamma_milli):
    st = hp.Stats()
    code = lib.hpeel_mphf_build_large(None, n, 1, gamma_milli, 1, None, None, ctypes.byref(st),
                                      None, 0, None, None)
    return code, lib.hpeel_last_error().decode()


# gamma small enough that a part's vertices still have 32-bit ids
@pytest.mark.parametrize("n", [1 << 39, (1 << 39) + 1, (1 << 40) - 1, 1 << 40])
def test_ids_past_the_id_sum_are_refused(lib, n):
    code, text = _call(lib, n, 1)
    assert code == 1 and "2^39" in text


def test_the_largest_id_width_is_not(lib):
    # refused too, for its NULL pointers or (no device here) for the device
    code, text = _call(lib, (1 << 39) - 1, 1)
    assert code != 0 and "2^39" not in text
