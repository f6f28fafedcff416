"""The work space eik_mlp_grad asks for: what its kernels write (one partial sum per parameter, and one of the squared
errors, for every 128 samples), at every size an int32_t can hold; a size it cannot is refused before the device is used."""
import ctypes as C

import pytest

from oracle import mlp


@pytest.fixture(scope="module")
def eik():
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as E
    return E


PER_BLOCK = mlp.n_params() + 1
MOST = (2 ** 31 - 1) // PER_BLOCK * 128


@pytest.mark.parametrize("B", [1, 127, 128, 129, 32768, 16646000, 16647000, 33294320, 66588640, MOST])
def test_size(eik, B):
    assert eik.eik_mlp_work_floats(B) == -(-B // 128) * PER_BLOCK


@pytest.mark.parametrize("B", [MOST + 1, 2 ** 31 - 1])
def test_too_many_samples_are_refused(eik, B):
    assert eik.eik_mlp_work_floats(B) == 0
    one = (C.c_float * 1)()
    p = C.cast(one, C.c_void_p)
    st = eik.lib().eik_mlp_grad(p, p, p, p, B, p, p, p, None)
    assert st == eik.EIK_EINVAL
