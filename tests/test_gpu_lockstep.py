"""Two cells of a warp take their attempts together (cells_per_warp = 2): a cell's result must not depend on its
partner.  Cells that end at different times, at once, with a bad input or with a singular or non-finite attempt
share warps with ordinary ones, in both launch forms, for odd and even counts; every ordinary cell must come out
bit for bit as it does alone (tolerance 0), and every other with its own status.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402


def _run(h, T, p, Y, dt, **kw):
    N = T.shape[0]
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    Tg, Yg, hio = d(T), d(Y), torch.zeros(N, dtype=torch.float64, device="cuda")
    ns, st = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    tr = torch.zeros(60, N, dtype=torch.float64, device="cuda")
    h.integrate(Tg, d(p), Yg, d(dt), hio, ns, st, trace=tr, cells_per_warp=2, max_substeps=400, **kw)
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (Tg, Yg, hio, ns, st, tr)]


@pytest.mark.parametrize("n_cells", [1, 2, 3, 16, 33])
@pytest.mark.parametrize("mode,chunk", [(0, 0), (1, 1), (1, 3)])
def test_results_do_not_depend_on_the_partner(n_cells, mode, chunk):
    m = synth.mechanism_small()
    h = chem.create(m, 0)
    F = synth.field_uniform_random(m, n_cells, seed=n_cells)
    rng = np.random.default_rng(n_cells)
    dt = 10.0 ** rng.uniform(-9, -6, n_cells)
    T, p, Y = F.T.copy(), F.p.copy(), F.Y.copy()
    kind = rng.integers(0, 8, n_cells)
    T[kind == 0] = -1.0            # bad input
    dt[kind == 1] = 0.0            # nothing to do
    p[kind == 2] = np.nan          # bad input
    T[kind == 3] = 1e9             # rates overflow: non-finite attempts
    dt[kind == 4] = 1e-2           # runs into max_substeps
    got = _run(h, T, p, Y, dt, mode=mode, chunk=chunk)
    for c in range(n_cells):
        one = _run(h, T[c:c + 1], p[c:c + 1], Y[:, c:c + 1], dt[c:c + 1], mode=0)
        for a, b in zip(got, one):
            assert np.array_equal(a[..., c:c + 1], b, equal_nan=True), (c, kind[c])
        assert got[4][c] == {0: 4, 2: 4}.get(int(kind[c]), got[4][c])
