"""A batch after a bounded wait gave up: sync reports it until the reset, which
restarts every chain (include/pcaden.h) and so must clear the flag that ends
every later wait.  The flag is set from here, on the stream's idle device: no
public call makes a batch's wait run out."""
import ctypes

import numpy as np
import pytest

from pcad_inputs import Model, gaussian_noise, greyscale_scene

pytestmark = pytest.mark.gpu

ETIMEOUT = 4


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


def _set_flag(pc, b):
    f = getattr(pc.lib(), "_ZN4pcad16batch_error_flagEP10pcad_batch")
    f.argtypes, f.restype = [ctypes.c_void_p], ctypes.c_void_p
    one = ctypes.c_int(1)
    cu = ctypes.CDLL("libcuda.so.1")
    assert cu.cuMemcpyHtoD_v2(ctypes.c_uint64(f(b)), ctypes.byref(one), ctypes.c_size_t(4)) == 0


def test_reset_recovers_a_batch_from_a_wait_that_gave_up(pc):
    m16 = Model(L=16, pair=1, pair_coef=0.6, pair_T=3, sigma=1.2, inertia=1.0)
    m33 = Model(L=33, nbhd=8, pair=0, pair_coef=0.8, sigma=3.0, inertia=0.4)   # wavefront items
    jobs = [(gaussian_noise(5, greyscale_scene(4, 150, 131, m.L, n_shapes=6), m.sigma, m.L), m, 3,
             i, 2) for i, m in enumerate((m16, m33))]
    b = pc.pcad_batch_create(jobs, autotune=False)
    try:
        pc.pcad_batch_set_tiling(b, 4, 2)
        pc.pcad_batch_run(b, 20)
        pc.pcad_batch_sync(b)
        want = [pc.pcad_batch_read_sample(b, i, *j[0].shape) for i, j in enumerate(jobs)]
        _set_flag(pc, b)
        for _ in range(2):
            with pytest.raises(pc.PcadError) as e:
                pc.pcad_batch_sync(b)
            assert e.value.status == ETIMEOUT
        pc.pcad_batch_reset(b)
        pc.pcad_batch_run(b, 20)
        pc.pcad_batch_sync(b)
        for i, j in enumerate(jobs):
            assert np.array_equal(pc.pcad_batch_read_sample(b, i, *j[0].shape), want[i])
    finally:
        pc.pcad_batch_destroy(b)
