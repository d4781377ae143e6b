"""The cell-pair stage kernel evaluates the traces across same-level and
outflow faces itself and takes level jumps and prescribed states from the
guard pass.  Every kind of block face at p = 1..3, through rotated frames and
with whole, ragged and single-layer z-chunks, against the oracle (p = 3 also
in the mortar mode) at the tolerances of test_gpu_parity, and bit for bit
between the chunk lengths and grids."""
import numpy as np
import pytest

import workloads as W
from oracle import dg
from oracle import forest as FO

from test_gpu_parity import TOL, assert_matches, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgf():
    import paper_2502_12620_gb300 as pkg
    pkg.lib()
    return pkg


def open_forest(jitter):
    """Two roots side by side without periodic gluing, the first refined once:
    same-level, coarser, finer and domain-boundary faces in rotated frames."""
    w = W.lattice_forest(3, (2, 1, 1), 1.0, 8, jitter=jitter, rotate_roots=True, seed=5, periodic=False)
    w["refine"] = [[(0, 1, (0, 0, 0))]]
    return w


@pytest.mark.parametrize("jitter", [0.0, 0.1])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_boundary_faces_match_oracle(dgf, p, jitter, monkeypatch):
    monkeypatch.setenv("DGF_STAGE_KERNEL", "pair")
    w = open_forest(jitter)
    f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP32, cfl=0.2)
    assert f.tuning()["stage_kernel"] == "pair"
    state = np.array([1.1, 0.2, -0.1, 0.05, 2.6])
    tags = np.zeros((2, 6), np.int32)
    tags[:, ::2] = 1  # prescribed state on the minus faces, outflow on the others
    f.set_boundary(tags, state)
    S = dg.Solver(FO.build(w), p, cfl=0.2, boundary=(tags, state))
    U = W.random_modal_state(f.n_leaves, 3, 8, p, seed=p).astype(np.float32).astype(np.float64)
    f.set_state(U)
    assert_matches(f.dg_residual(), S.residual(U), "fp32", S, U)
    f.close()


@pytest.mark.parametrize("mode", ["paper", "mortar"])
def test_p3_residual_and_step_match_oracle(dgf, mode, monkeypatch):
    monkeypatch.setenv("DGF_STAGE_KERNEL", "pair")
    w = W.lattice_forest(3, (2, 1, 1), 1.0, 8, jitter=0.1, rotate_roots=True, seed=3)
    w["refine"] = [[(0, 1, (0, 0, 0))]]
    f = dgf.Forest.from_workload(w, p=3, precision=dgf.FP32, cfl=0.2, nonconforming=mode)
    assert f.tuning()["stage_kernel"] == "pair"
    S = dg.Solver(FO.build(w), 3, cfl=0.2, nonconforming=mode)
    U = W.random_modal_state(f.n_leaves, 3, 8, 3, seed=30).astype(np.float32).astype(np.float64)
    f.set_state(U)
    assert_matches(f.dg_residual(), S.residual(U), "fp32", S, U)
    f.rk_step()
    assert rel(f.get_state(), S.ssp_rk3_step(U, S.dt(U))) < TOL["fp32"]
    assert f.status_word() == 0
    f.close()


@pytest.mark.parametrize("jitter", [0.0, 0.1])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_chunks_and_grids_change_no_bit(dgf, p, jitter, monkeypatch):
    monkeypatch.setenv("DGF_STAGE_KERNEL", "pair")
    out = []
    for z, grid in ((8, "persistent"), (8, "items"), (3, "items"), (1, "persistent")):
        monkeypatch.setenv("DGF_ZCHUNK", str(z))
        monkeypatch.setenv("DGF_STAGE_GRID", grid)
        f = dgf.Forest.from_workload(open_forest(jitter), p=p, precision=dgf.FP32, cfl=0.2)
        f.set_state(W.random_modal_state(f.n_leaves, 3, 8, p, seed=2).astype(np.float32))
        R = f.dg_residual()
        f.run(3)
        out.append((R, f.get_state()))
        assert f.status_word() == 0
        f.close()
    for R, U in out[1:]:
        assert np.array_equal(R, out[0][0]) and np.array_equal(U, out[0][1])
