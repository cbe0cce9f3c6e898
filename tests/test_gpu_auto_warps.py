"""The library's own choice of lanes per cell, for mechanisms between and at the sizes of the other tests: two warps where
fewer than six one-warp cells fit an SM, whatever number of two-warp cells the kernels' registers allow (four; five
one-warp cells of 39 to 46 KB fit).  A default call must return what the call with that choice spelt out returns, bit for
bit (tolerance 0).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402


def _between(n, R, core_frac):
    return synth.make_mechanism(9, n, R, R // 10, R // 15, ["C", "H", "O", "N"], {"C": 3, "H": 8, "O": 3, "N": 2}, 9,
                                fuel={"C": 1, "H": 4}, core_frac=core_frac)


def _run(h, F, **kw):
    N = F.n_cells
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    Tg, Yg, hio = d(F.T), d(F.Y), torch.zeros(N, dtype=torch.float64, device="cuda")
    ns, st = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    h.integrate(Tg, d(F.p), Yg, d(F.dt), hio, ns, st, **kw)
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (Tg, Yg, hio, ns, st)]


@pytest.mark.parametrize("mech,fits,warps", [
    ((90, 600, 0.06), 5, 2), ((90, 600, 0.08), 5, 2), ((100, 650, 0.06), 5, 2), ((90, 600, 0.12), 4, 2),
    (synth.mechanism_large, 3, 2), (synth.mechanism_methane_sized, 6, 1)])
def test_default_call_takes_the_documented_choice(mech, fits, warps):
    m = mech() if callable(mech) else _between(*mech)
    h = chem.create(m, 0)
    F = synth.field_uniform_random(m, 24, seed=5, dt=1e-8)
    for mode in (0, 1):
        a, b = _run(h, F, mode=mode), _run(h, F, mode=mode, warps_per_cell=warps)
        assert min(h.info["resident_cells"][0], 6) == fits and h.info["auto_warps_per_cell"] == warps
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
