"""Where the library's launch choice changes with the number of cells: kernels with helper warps, and one or two warps per
cell in the reverse pass of the adjoint.  The counts at which it changes are found by asking the library
(chem_launch_shape), so the runs compared on either side are known to take different kernels.

Neither choice may change a bit of a result (tolerance 0): helper warps only evaluate reactions, and the reverse pass adds
the same terms in the same order with one warp as with two, so that a cell's gradient does not depend on how a field is
split over calls.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402
from tests.test_gpu_adjoint_warps import MECH, _adjoint  # noqa: E402
from tests.test_gpu_helpers import _run  # noqa: E402


def _most(h, holds, **opts):
    """The largest number of cells for which holds(launch shape) is true (0: none); it is false beyond."""
    lo, hi = 0, 1 << 16
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if holds(h.launch_shape(mid, **opts)) else (lo, mid)
    return lo


@pytest.mark.parametrize("mech,wpc,forms", [("methane", 1, (3, 1)), ("methane", 2, (2,)), ("large", 1, (3, 1)),
                                            ("large", 2, (2,)), ("small", 1, ())])
def test_helpers_up_to_where_all_cells_fit(mech, wpc, forms):
    m = MECH[mech]()
    h = chem.create(m, 0)
    opts = dict(warps_per_cell=wpc, cells_per_warp=1)
    edges = {f: _most(h, lambda s: s["helper_warps"] >= f, **opts) for f in forms}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert all(e > 0 and e % sms == 0 for e in edges.values())
    assert h.launch_shape(1, **opts)["helper_warps"] == (forms[0] if forms else 0)
    for form, edge in edges.items():
        for N in (edge, edge + 1):
            assert (h.launch_shape(N, **opts)["helper_warps"] >= form) == (N == edge)
            assert h.launch_shape(N, block_cells=1, **opts)["helper_warps"] == 0
            F = synth.field_uniform_random(m, N, seed=N)
            dt = 10.0 ** np.random.default_rng(N).uniform(-9, -7.5, N)
            for mode in (0, 1):
                a = _run(h, F.T, F.p, F.Y, dt, mode=mode, max_substeps=40, **opts)
                b = _run(h, F.T, F.p, F.Y, dt, mode=mode, max_substeps=40, block_cells=1, **opts)
                for x, y in zip(a, b):
                    assert np.array_equal(x, y, equal_nan=True)


@pytest.mark.parametrize("mech,n_cells,dt", [("small", 7, 1e-7), ("methane", 33, 2e-7), ("large", 5, 2e-8)])
def test_reverse_pass_where_two_warps_no_longer_fit(mech, n_cells, dt):
    m = MECH[mech]()
    h = chem.create(m, 0)
    edge = _most(h, lambda s: s["adjoint_warps"] == 2)
    assert edge >= n_cells and h.launch_shape(edge + 1)["adjoint_warps"] == 1
    F = synth.field_uniform_random(m, n_cells, seed=n_cells, dt=dt)
    rng = np.random.default_rng(n_cells)
    gT, gY = rng.standard_normal(n_cells) * 1e-3, rng.standard_normal((m.n_species, n_cells))
    rep = np.arange(edge + 1) % n_cells
    one = _adjoint(h, F.T[rep], F.p[rep], F.Y[:, rep], F.dt[rep], gT[rep], gY[:, rep])
    two = _adjoint(h, F.T, F.p, F.Y, F.dt, gT, gY)
    for a, b in zip(two, one):
        assert np.array_equal(a, b[..., :n_cells], equal_nan=True)
