"""2D stage tiles: forests too small to fill the GPU sweep their blocks in
slabs of a quarter of the rows, larger ones block by block (n_seg = 2 always).
Both against the oracle, on either side of the line, in the paper and mortar
level-jump modes, at the tolerances of test_gpu_parity."""
import numpy as np
import pytest

import workloads as W
from oracle import dg
from oracle import forest as FO

from test_gpu_parity import TOL, assert_matches, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["paper", "mortar"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("B,n,p", [(12, 4, 1), (13, 4, 2), (13, 2, 3), (3, 8, 3)])
def test_2d_tiles_match_oracle(B, n, p, prec, mode):
    import paper_2502_12620_gb300 as dgf
    w = W.lattice_forest(2, B, 1.0, n, jitter=0.1, rotate_roots=True, seed=B)
    w["refine"] = [[(0, 1, (0, 0))]]
    f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP64 if prec == "fp64" else dgf.FP32, cfl=0.2,
                                 nonconforming=mode)
    S = dg.Solver(FO.build(w), p, cfl=0.2, nonconforming=mode)
    U = W.random_modal_state(f.n_leaves, 2, n, p, seed=p).astype(f.dtype).astype(np.float64)
    f.set_state(U)
    assert_matches(f.dg_residual(), S.residual(U), prec, S, U)
    f.rk_step()
    assert rel(f.get_state(), S.ssp_rk3_step(U, S.dt(U))) < TOL[prec]
    f.close()
