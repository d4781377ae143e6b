"""What the first time step of a forest picks: stage kernel, chunk length, grid."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgf():
    import paper_2502_12620_gb300 as pkg
    pkg.lib()
    return pkg


def forest(dgf, w, p, mode):
    f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP32, cfl=0.05, nonconforming=mode)
    f.project(W.smooth_state)
    f.run(5)
    return f


def test_choice_does_not_outlive_a_pin(dgf, monkeypatch):
    """A forest tuned with a pinned kernel, chunk or grid leaves the free
    choice of the next one of its shape alone."""
    w = W.periodic_cube_forest(3)
    monkeypatch.setenv("DGF_STAGE_KERNEL", "classic")
    monkeypatch.setenv("DGF_ZCHUNK", "3")
    f = forest(dgf, w, 2, "paper")
    assert f.tuning()["zchunk"] == 3 and f.tuning()["stage_kernel"] == "classic"
    f.close()
    monkeypatch.delenv("DGF_STAGE_KERNEL")
    monkeypatch.delenv("DGF_ZCHUNK")
    f = forest(dgf, w, 2, "paper")
    assert f.tuning()["zchunk"] in (1, 2, 4, 8)
    f.close()
