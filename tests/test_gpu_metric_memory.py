"""The metric tables of FP64 forests with curved blocks are a convenience of
the stage kernel: where they do not fit beside what a forest needs they are
given up, not the state."""
import pytest

import workloads as W

from test_gpu_parity import TOL, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgf():
    import paper_2502_12620_gb300 as pkg
    pkg.lib()
    return pkg


def met_bytes(w, p, leaves):
    """Size of the first table; where it is refused the second is not asked for."""
    d, N = w["dim"], p + 1
    return leaves * w["n_seg"] ** d * (d * d + 1) * N ** d * 8


class _Limited:
    """The binding's allocator with a bound on the bytes held and a test for
    refused sizes; records the most bytes held."""

    def __init__(self, dgf, base, limit, refuse):
        self.base, self.struct, self.peak, self.refused = base, base.struct, 0, 0
        plain = base._a

        def alloc(ctx, nbytes, stream):
            if nbytes in refuse or sum(base.live.values()) + nbytes > limit:
                self.refused += 1
                return None
            q = plain(ctx, nbytes, stream)
            self.peak = max(self.peak, sum(base.live.values()))
            return q

        self._alloc = dgf._ALLOC_FN(alloc)
        self.struct = dgf._Allocator(None, self._alloc, base._f)

    @property
    def live(self):
        return self.base.live


@pytest.mark.parametrize("d,p", [(2, 3), (3, 1), (3, 2)])
def test_regrid_in_the_memory_of_a_forest_without_tables(dgf, d, p, monkeypatch):
    """A march through a refinement and a coarsening, once with the tables'
    allocations refused and then within the most bytes that this one held:
    the tables fit there at times, but not beside a regrid's buffers."""
    w = W.lattice_forest(d, (2,) + (1,) * (d - 1), 1.0, 4, jitter=0.1, rotate_roots=True, seed=4)
    base = dgf._TorchAllocator
    refuse = {met_bytes(w, p, leaves) for leaves in (2, 1 + 2 ** d)}
    made = []

    def march(limit, refused):
        def make(device):
            made.append(_Limited(dgf, base(device), limit, refused))
            return made[-1]

        monkeypatch.setattr(dgf, "_TorchAllocator", make)
        f = dgf.Forest.from_workload(w, p=p, precision=dgf.FP64, cfl=0.1)
        f.project(W.smooth_state)
        f.run(2)
        f.refine([0])
        f.run(2)
        f.fill_guardcells()
        f.run(1)
        f.coarsen(list(range(2 ** d)))
        f.run(2)
        U = f.get_state()
        assert f.status_word() == 0
        f.close()
        return U, made[-1]

    U0, a0 = march(1 << 40, refuse)
    assert a0.refused > 0
    U1, a1 = march(a0.peak, ())
    assert a1.refused > 0 and a1.peak <= a0.peak
    # the metric from tables or evaluated in place: rounding only
    assert rel(U1, U0) < TOL["fp64"]
    U2, a2 = march(1 << 40, ())
    assert a2.refused == 0 and rel(U2, U0) < TOL["fp64"]
