"""Single-channel convolutions of more than 2^30 output pixels are refused (the limit the header
states), on every kernel that would take them: before any device call, so that no device is
needed and nothing runs."""
import ctypes

import pytest

from paper_1911_00357_gb300 import binding as B

E_CONFIG = -2


def _conv(N, H, W, k, s, p, Cout):
    q = ctypes.c_void_p(256)  # never read: the call is refused
    return B.lib().ddppo_conv2d(N, H, W, 1, Cout, k, s, p, q, q, q, ctypes.c_float(0.0), None, None)


@pytest.mark.parametrize("N,H,k,s,p,Cout", [(262145, 128, 7, 2, 3, 32), (262145, 128, 7, 2, 3, 64),
                                            (66000, 128, 8, 1, 4, 16), (70000, 256, 7, 2, 3, 32)])
def test_too_many_output_pixels_are_refused(N, H, k, s, p, Cout):
    assert N * ((H + 2 * p - k) // s + 1) ** 2 > 1 << 30
    assert _conv(N, H, H, k, s, p, Cout) == E_CONFIG
    B.lib().ddppo_last_error.restype = ctypes.c_char_p
    assert b"2^30" in B.lib().ddppo_last_error()
