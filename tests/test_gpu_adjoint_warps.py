"""The reverse pass with two warps per cell (few cells) against the pass with one (more cells than fit at once): the
same cells, alone and repeated past the change.  Both add the same terms to the state's adjoint in the same order, so
final states and initial-state gradients must agree bit for bit.  The parameter gradients are two sums over the steps
instead of one: with up to 4,096 steps of 4 contributions the order of additions moves a sum by at most 2^14 x 2^-53 =
2e-12 of the sum of its terms' magnitudes, held here to 1e-10 of the cell's largest gradient.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402

MECH = {"small": synth.mechanism_small, "methane": synth.mechanism_methane_sized, "large": synth.mechanism_large}


def _adjoint(h, T, p, Y, dt, gT, gY):
    N = T.shape[0]
    d = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")
    Tg, Yg, gA, gE, gc, gT0, gY0 = d(T), d(Y), z(h.R), z(h.R), z(2 * h.R, N), z(N), z(h.n, N)
    st = torch.zeros(N, dtype=torch.int32, device="cuda")
    h.adjoint(Tg, d(p), Yg, d(dt), d(gT), d(gY), gA, gE, st, grad_cell=gc, gT0=gT0, gY0=gY0, tape_steps=96)
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (Tg, Yg, gT0, gY0, st, gc)]


@pytest.mark.parametrize("mech,n_cells,many,dt", [("small", 1, 2600, 1e-8), ("small", 7, 2600, 1e-7),
                                                  ("methane", 1, 620, 1e-8), ("methane", 33, 620, 3e-8),
                                                  ("large", 5, 160, 3e-9)])
def test_two_warps_per_cell_match_one(mech, n_cells, many, dt):
    m = MECH[mech]()
    h = chem.create(m, 0)
    F = synth.field_uniform_random(m, n_cells, seed=n_cells, dt=dt)
    rng = np.random.default_rng(n_cells)
    T, p, Y, dtc = F.T.copy(), F.p.copy(), F.Y.copy(), F.dt.copy()
    if n_cells > 4:
        dtc[1] = 0.0     # no step
        dtc[3] = 1e-5    # more steps than the tape holds
        T[2] = -1.0      # bad input
    gT, gY = rng.standard_normal(n_cells) * 1e-3, rng.standard_normal((m.n_species, n_cells))
    rep = np.arange(many) % n_cells
    one = _adjoint(h, T[rep], p[rep], Y[:, rep], dtc[rep], gT[rep], gY[:, rep])
    two = _adjoint(h, T, p, Y, dtc, gT, gY)
    for a, b in zip(two[:5], one[:5]):
        assert np.array_equal(a, b[..., :n_cells], equal_nan=True)
    for c in range(n_cells):
        a, b = two[5][:, c], one[5][:, c]
        for half in (slice(0, h.R), slice(h.R, 2 * h.R)):
            assert np.max(np.abs(a[half] - b[half])) <= 1e-10 * np.max(np.abs(b[half])), c
