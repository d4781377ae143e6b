"""State hand-over (dgf_set_state / dgf_get_state): the conversion between the
modal interface layout and the nodal state buffer, from and to host arrays,
device tensors and device addresses that are not aligned to an element (those
take the staged copy), and the CFL minimum taken on the way in.

A modal -> nodal -> modal round trip of N-point transforms along d axes: each
of the 2 d passes sums at most N + 1 rounded terms whose absolute sum is at
most 3 N times the cell's largest value (|V|, |Vi| rows), so the relative
error of a cell stays below 2 d (N + 2) (3 N)^2 eps.
"""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgf():
    import paper_2502_12620_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_comp"])
@pytest.mark.parametrize("p", [0, 1, 2, 3])
@pytest.mark.parametrize("dim,n", [(2, 2), (2, 8), (3, 2), (3, 4)])
def test_state_round_trip_and_cfl(dgf, dim, n, p, prec):
    import torch
    w = W.rotated_pair_2d(n_seg=n) if dim == 2 else W.jitter3d_forest(seed=2, n_seg=n)
    pr = {"fp64": dgf.FP64, "fp32": dgf.FP32, "fp32_comp": dgf.FP32_COMP}[prec]
    f = dgf.Forest.from_workload(w, p=p, precision=pr, cfl=0.2)
    U = W.random_modal_state(f.n_leaves, dim, n, p, seed=p).astype(f.dtype)
    dev = torch.from_numpy(U).cuda()
    tol = 2 * dim * (p + 3) * (3 * (p + 1)) ** 2 * np.finfo(f.dtype).eps * np.abs(U).max()

    f.set_state(U)
    host = f.get_state()
    assert np.abs(host.astype(float) - U).max() <= tol
    dt = f.rk_step(return_dt=True)
    f.set_state(dev)
    out = torch.empty_like(dev)
    assert np.array_equal(f.get_state(out).cpu().numpy(), host) and np.array_equal(f.get_state(), host)
    assert f.rk_step(return_dt=True) == dt
    # the CFL minimum of the hand-over is the one of the CFL kernel
    f.set_state(dev)
    assert f.compute_dt() == dt

    # addresses off the element grid keep the staged copy
    raw = torch.zeros(U.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[1:1 + U.nbytes] = dev.view(torch.uint8).flatten()
    torch.cuda.synchronize()
    L = dgf.lib()
    assert L.dgf_set_state(f.h, ctypes.c_void_p(raw.data_ptr() + 1), 1) == 0
    assert np.array_equal(f.get_state(), host)
    raw.zero_()
    torch.cuda.synchronize()
    assert L.dgf_get_state(f.h, ctypes.c_void_p(raw.data_ptr() + 3), 1) == 0
    got = raw[3:3 + U.nbytes].cpu().numpy().tobytes()
    assert got == np.ascontiguousarray(host).tobytes()
    f.close()
