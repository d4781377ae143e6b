"""Finer-neighbour guard cells in number: beyond about 2,400 of them the guard
pass gives a cell to a warp instead of a block.  Nine of 27 roots refined make
some 50 such faces of 64 cells; curved blocks (an operator per guard cell) in
rotated frames and affine ones (a shared operator), against the oracle at the
tolerances of test_gpu_parity."""
import numpy as np
import pytest

import workloads as W
from oracle import dg
from oracle import forest as FO

from test_gpu_parity import assert_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,p,jitter", [("fp32", 1, 0.1), ("fp32", 2, 0.0), ("fp64", 1, 0.1), ("fp32_comp", 1, 0.0)])
def test_many_finer_faces_match_oracle(prec, p, jitter):
    import paper_2502_12620_gb300 as dgf
    w = W.lattice_forest(3, 3, 1.0, 8, jitter=jitter, rotate_roots=True, seed=9)
    w["refine"] = [[(r, 1, (0, 0, 0)) for r in range(27) if (r % 3 + r // 3 % 3 + r // 9) % 3 == 0]]
    f = dgf.Forest.from_workload(w, p=p, precision={"fp32": dgf.FP32, "fp64": dgf.FP64, "fp32_comp": dgf.FP32_COMP}[prec])
    assert int((f.leaf_table()["kind"] == dgf.FINER).sum()) * 64 > 2432
    S = dg.Solver(FO.build(w), p)
    U = W.random_modal_state(f.n_leaves, 3, 8, p, seed=4).astype(np.float32).astype(np.float64)
    f.set_state(U)
    assert_matches(f.dg_residual(), S.residual(U), prec, S, U)
    f.close()
