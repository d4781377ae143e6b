"""A device buffer whose allocation ends before the state does is refused by
the hand-over (kernels read and write callers' buffers in place), and the
forest's state stays."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

IPC_CAPABLE = 10  # CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE


@pytest.fixture(scope="module")
def dgf():
    import paper_2502_12620_gb300 as pkg
    pkg.lib()
    return pkg


def bytes_behind(t):
    """Bytes from a tensor's address to the end of its cudaMalloc allocation
    (None where the allocation is not one cudaMalloc)."""
    cu = ctypes.CDLL("libcuda.so.1")
    p = ctypes.c_uint64(t.data_ptr())
    whole, base, size = ctypes.c_uint64(0), ctypes.c_uint64(0), ctypes.c_size_t(0)
    if cu.cuPointerGetAttribute(ctypes.byref(whole), IPC_CAPABLE, p) or not whole.value:
        return None
    if cu.cuMemGetAddressRange_v2(ctypes.byref(base), ctypes.byref(size), p):
        return None
    return base.value + size.value - p.value


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_comp"])
def test_short_device_buffers_are_refused(dgf, prec):
    import torch
    pr = {"fp64": dgf.FP64, "fp32": dgf.FP32, "fp32_comp": dgf.FP32_COMP}[prec]
    f = dgf.Forest.from_workload(W.periodic_cube_forest(3), p=2, precision=pr)
    U = W.random_modal_state(f.n_leaves, 3, 8, 2, seed=1).astype(f.dtype)
    f.set_state(U)
    host = f.get_state()
    short = torch.zeros(8, dtype=torch.float64, device="cuda")
    room = bytes_behind(short)
    if room is None or room >= U.nbytes:
        pytest.skip("the allocation behind a small tensor is not known to be short")
    torch.cuda.synchronize()
    for call in (lambda: f.get_state(short),
                 lambda: dgf._check(dgf.lib().dgf_set_state(f.h, ctypes.c_void_p(short.data_ptr()), 1))):
        with pytest.raises(dgf.DgfError) as e:
            call()
        assert dgf.STATUS[e.value.code] == "EINVAL"
    assert np.array_equal(f.get_state(), host) and not short.any().item()
    f.rk_step()
    assert f.status_word() == 0
    f.close()
