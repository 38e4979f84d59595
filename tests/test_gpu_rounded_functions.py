"""recip, root, third and recip_sqrt of the step kernels against CUDA's rounded
division and square root, for every significand at every exponent of the range
that their comments state (the steps on 16-bit storage and with a symmetry axis
are reproduced to the last bit on the strength of it).

recip_sqrt is not rounded correctly: a Newton step on an approximation good to
2^-22 leaves its own rounding (2^-24 of the result at most) and half of that of
the product x r in its residual, 1.5 x 2^-24; the rounded reciprocal of the
rounded root, which it stands for, has the same bound."""
import ctypes

import numpy as np
import pytest

import device_functions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    return device_functions.load(tmp_path_factory.mktemp("device_functions"))


@pytest.mark.parametrize("fn,lowest,highest,negative", [(0, -126, 125, 0), (0, -126, 125, 1), (1, -102, 127, 0),
                                                        (2, -122, 127, 0), (2, -122, 127, 1)],
                         ids=["recip", "recip-negative", "root", "third", "third-negative"])
def test_rounded_for_every_significand(functions, fn, lowest, highest, negative):
    bad = np.zeros(highest - lowest + 1, np.uint32)
    assert functions.scan_rounded(fn, lowest, len(bad), negative, bad.ctypes.data_as(ctypes.c_void_p)) == 0
    assert not bad.any(), [(lowest + int(k), int(bad[k])) for k in np.nonzero(bad)[0]]


def test_recip_sqrt_is_no_further_off_than_the_rounded_root(functions):
    worst = np.zeros(2, np.float32)
    # squared gradients: held above 1e-8 (2^-27), at most about 1
    assert functions.scan_recip_sqrt(-27, 40, worst.ctypes.data_as(ctypes.c_void_p)) == 0
    assert worst[0] <= 1.5 and worst[0] <= worst[1]
