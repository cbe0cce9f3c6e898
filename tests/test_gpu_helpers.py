"""Calls with few cells run on kernels whose cells have helper warps for the reaction rounds.  A reaction's results do
not depend on the lane that evaluates it, so these kernels must return what the kernels without helpers return, bit
for bit (tolerance 0): states, steps, counts, status and step trace, at the cell counts where the choice changes, in
both launch forms, for all methods, with tabulated functions, and for cells that end without an attempt, fail or run
into the attempt limit.  A given block_cells selects the kernels without helpers.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402

MECH = {"methane": synth.mechanism_methane_sized, "large": synth.mechanism_large, "small": synth.mechanism_small}
SMS = 152


def _run(h, T, p, Y, dt, **kw):
    N = T.shape[0]
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    Tg, Yg, hio = d(T), d(Y), torch.zeros(N, dtype=torch.float64, device="cuda")
    ns, st = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    tr = torch.zeros(40, N, dtype=torch.float64, device="cuda")
    h.integrate(Tg, d(p), Yg, d(dt), hio, ns, st, trace=tr, **kw)
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (Tg, Yg, hio, ns, st, tr)]


@pytest.mark.parametrize("mech,wpc,n_cells,mode,kw", [
    ("methane", 1, 1, 0, {}), ("methane", 1, 31, 1, {}), ("methane", 1, 2 * SMS, 0, {}), ("methane", 1, 2 * SMS + 1, 1, {}),
    ("methane", 1, 4 * SMS, 1, {}), ("methane", 1, 4 * SMS + 1, 0, {}), ("methane", 2, 65, 0, {}),
    ("methane", 1, 77, 0, dict(method=1)), ("methane", 1, 400, 1, dict(method=2)), ("methane", 1, 60, 1, dict(tabulate=1)),
    ("large", 2, 9, 1, {}), ("large", 2, 2 * SMS + 1, 0, {}), ("large", 1, 40, 0, {}), ("small", 1, 50, 0, {})])
def test_helpers_change_no_bit(mech, wpc, n_cells, mode, kw):
    m = MECH[mech]()
    h = chem.create(m, 0)
    F = synth.field_uniform_random(m, n_cells, seed=n_cells)
    rng = np.random.default_rng(n_cells)
    dt = 10.0 ** rng.uniform(-9, -7, n_cells)
    T, p, Y = F.T.copy(), F.p.copy(), F.Y.copy()
    if n_cells > 8:
        kind = rng.integers(0, 16, n_cells)
        T[kind == 0] = -1.0            # bad input
        dt[kind == 1] = 0.0            # nothing to do
        p[kind == 2] = np.nan          # bad input
        T[kind == 3] = 1e9             # rates overflow: non-finite attempts
        dt[kind == 4] = 1e-2           # runs into max_substeps
    a = _run(h, T, p, Y, dt, mode=mode, warps_per_cell=wpc, cells_per_warp=1, max_substeps=60, **kw)
    b = _run(h, T, p, Y, dt, mode=mode, warps_per_cell=wpc, cells_per_warp=1, max_substeps=60, block_cells=1, **kw)
    for x, y in zip(a, b):
        assert np.array_equal(x, y, equal_nan=True)
