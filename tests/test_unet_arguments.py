"""Pointers that no convolution kernel could load or store are refused on the host, before any
launch (the calls below never reach a device)."""
import ctypes

import pytest

from paper_2003_11069_gb300 import lbnci, unet

BASE = 1 << 20  # stands for a 256-byte aligned device address; nothing reads it


def _conv(x=0, w=0, y=0):
    p = [ctypes.c_void_p(BASE + o) for o in (x, w, y)]
    return unet.load().lbu_conv3x3(p[0], 32, 1, 8, 8, 32, 0, p[1], None, 0, p[2], 32, 32, None)


def _wgrad(x=0, dy=0, work=0):
    p = [ctypes.c_void_p(BASE + o) for o in (x, dy, work)]
    n = unet.conv3x3_wgrad_work(1, 8, 8, 32, 32)
    return unet.load().lbu_conv3x3_wgrad(p[0], 32, 1, 8, 8, 32, 0, p[1], 32, 32, ctypes.c_void_p(BASE), None, p[2], n,
                                         None)


@pytest.mark.parametrize("call", [lambda: _conv(x=2), lambda: _conv(x=8), lambda: _conv(w=4), lambda: _conv(w=8),
                                  lambda: _conv(y=2), lambda: _wgrad(x=8), lambda: _wgrad(dy=2), lambda: _wgrad(dy=8),
                                  lambda: _wgrad(work=4)])
def test_misaligned_operands_are_refused(call):
    assert call() == lbnci.LB_EINVAL
    assert b"alignment" in unet.load().lbu_last_error(None)
