"""The allocation-free entry point refuses meshes beyond its fixed scratch array, whichever of the solves a call asks for
(a refused call returns before any CUDA call, so this needs no GPU)."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2103_03407_gb300 import build

    return C.CDLL(build.build())


@pytest.mark.parametrize("prec,nf,nc,np_,fine,prev", [(0, 512, 32, 0, True, False), (0, 512, 256, 256, True, True),
                                                     (0, 512, 32, 32, False, True), (1, 1024, 32, 0, True, False),
                                                     (1, 1024, 32, 32, False, True), (1, 4096, 4096, 4096, False, True)])
def test_meshes_beyond_the_array_are_refused(lib, prec, nf, nc, np_, fine, prev):
    p = C.c_void_p(256)  # never read
    f = lib.mq_twogrid_samples_noalloc
    f.argtypes = [C.c_int32] * 5 + [C.c_void_p] * 3 + [C.c_double] + [C.c_void_p] * 4
    assert f(nf, nc, np_, prec, 1, p if fine else None, p, p if prev else None, 0.0, p, p, p, None) == 1
