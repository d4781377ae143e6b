"""Forests that hold affine and curved blocks together: the cell-pair stage
kernel copies geometry rows for the curved ones only, and one CTA of its
persistent grid sweeps blocks of both kinds in turn.  Against the oracle on a
small forest at the tolerances of test_gpu_parity, and bit for bit between
every chunk length and grid on one with more work items than resident CTAs."""
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


def mixed_forest(roots):
    """A lattice of rotated roots, the first refined; every third root, the
    first among them, has its inner cell nodes moved (its faces stay planar)
    and so consists of curved blocks, the others of affine ones."""
    w = W.lattice_forest(3, roots, 1.0, 8, rotate_roots=True, seed=11)
    rng = np.random.default_rng(12)
    for r in range(0, len(w["root_corners"]), 3):
        x = w["root_cell_nodes"][r].reshape(9, 9, 9, 3).copy()
        h = np.min(1.0 / (8 * np.asarray(roots)))
        x[1:-1, 1:-1, 1:-1] += rng.uniform(-0.1 * h, 0.1 * h, x[1:-1, 1:-1, 1:-1].shape)
        w["root_cell_nodes"][r] = x.reshape(-1, 3)
    w["refine"] = [[(0, 1, (0, 0, 0))]]
    return w


@pytest.mark.parametrize("mode", ["paper", "mortar"])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_mixed_forest_matches_oracle(dgf, p, mode, monkeypatch):
    monkeypatch.setenv("DGF_STAGE_KERNEL", "pair")
    w = mixed_forest((2, 2, 1))
    f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP32, cfl=0.2, nonconforming=mode)
    assert f.tuning()["stage_kernel"] == "pair"
    S = dg.Solver(FO.build(w), p, cfl=0.2, nonconforming=mode)
    U = W.random_modal_state(f.n_leaves, 3, 8, p, seed=p).astype(np.float32).astype(np.float64)
    f.set_state(U)
    assert_matches(f.dg_residual(), S.residual(U), "fp32", S, U)
    f.rk_step()
    assert rel(f.get_state(), S.ssp_rk3_step(U, S.dt(U))) < TOL["fp32"]
    assert f.status_word() == 0
    f.close()


@pytest.mark.parametrize("mode", ["paper", "mortar"])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_mixed_forest_chunks_and_grids_change_no_bit(dgf, p, mode, monkeypatch):
    """157 leaves on at most 456 resident CTAs at p = 1, 71 on 152 at p = 2, 3:
    more items than CTAs from three-layer chunks down.  One CTA per whole block
    is the tiling in which no CTA meets a second item.  At p = 1 both CTA
    shapes."""
    w = mixed_forest((6, 5, 5) if p == 1 else (4, 4, 4))
    U = W.random_modal_state(157 if p == 1 else 71, 3, 8, p, seed=2).astype(np.float32)

    def result():
        f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP32, cfl=0.2, nonconforming=mode)
        f.set_state(U)
        R = f.dg_residual()
        f.run(2)
        out = R, f.get_state()
        assert f.status_word() == 0
        f.close()
        return out

    monkeypatch.setenv("DGF_STAGE_KERNEL", "pair")
    monkeypatch.setenv("DGF_ZCHUNK", "8")
    monkeypatch.setenv("DGF_STAGE_GRID", "items")
    R0, U0 = result()
    for kernel in ("pair", "pair5") if p == 1 else ("pair",):
        monkeypatch.setenv("DGF_STAGE_KERNEL", kernel)
        for z in (8, 4, 3, 2, 1):
            for grid in ("persistent", "items"):
                monkeypatch.setenv("DGF_ZCHUNK", str(z))
                monkeypatch.setenv("DGF_STAGE_GRID", grid)
                R, U1 = result()
                assert np.array_equal(R, R0) and np.array_equal(U1, U0), (kernel, z, grid)
    # tuned freely: every tiling is timed on the way; whichever kernel is taken
    # (each is within TOL of the oracle)
    for k in ("DGF_STAGE_KERNEL", "DGF_ZCHUNK", "DGF_STAGE_GRID"):
        monkeypatch.delenv(k)
    R, U1 = result()
    assert rel(R, R0) < 2 * TOL["fp32"] and rel(U1, U0) < 2 * TOL["fp32"]
