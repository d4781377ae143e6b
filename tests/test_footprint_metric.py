"""The footprint estimate of a solve counts the metric tables that FP64
forests with curved blocks hold."""
import pytest

import workloads as W
from paper_2502_12620_gb300 import FP32, FP32_COMP, FP64
from paper_2502_12620_gb300.serve import footprint_bytes, leaf_count


def table_bytes(w, p, leaves=None):
    d, N = w["dim"], p + 1
    cells = (leaf_count(w) if leaves is None else leaves) * w["n_seg"] ** d
    return cells * (d * d + 1) * N ** d * 8, cells * d * d * N ** (d - 1) * 8


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("p", [0, 1, 2, 3])
def test_footprint_counts_metric_tables(d, p):
    flat = W.lattice_forest(d, 2, 1.0, 8, rotate_roots=True, seed=1)
    curved = W.lattice_forest(d, 2, 1.0, 8, rotate_roots=True, jitter=0.1, seed=1)
    trapezoid = dict(flat, root_cell_nodes=None, nodes=flat["nodes"] + 0.1 * flat["nodes"][:, :1] * flat["nodes"][:, 1:2])
    assert footprint_bytes(dict(flat, root_cell_nodes=None), p, FP64) == footprint_bytes(flat, p, FP64)
    for w in (curved, trapezoid):
        assert footprint_bytes(w, p, FP64) - footprint_bytes(flat, p, FP64) == sum(table_bytes(w, p))
        for prec in (FP32, FP32_COMP):
            assert footprint_bytes(w, p, prec) == footprint_bytes(flat, p, prec)


@pytest.mark.gpu
@pytest.mark.parametrize("p", [1, 2])
def test_footprint_of_curved_fp64_matches_allocation(p):
    import paper_2502_12620_gb300 as dgf
    w = W.jitter3d_forest(seed=0)
    f = dgf.Forest.from_workload(w, p=p, precision=FP64)
    f.project(W.smooth_state)
    f.rk_step()
    actual, est = f.device_bytes, footprint_bytes(w, p, FP64)
    f.close()
    assert 0.8 * actual < est < 1.25 * actual, (est, actual)
