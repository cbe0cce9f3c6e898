"""The elimination and substitution programs as the device runs them (rescheduled, in blocks of steps), through a
short integration against the oracle, for factor sizes around the lane groups' widths: with fewer unknowns than
lanes, as many, one more, and programs shorter than a block.  Each method and lane group; T and Y within 1e-8.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.oracle import Oracle  # noqa: E402
from paper_2311_14941_gb300 import chem  # noqa: E402
from tests import tinymech as tm  # noqa: E402


def _chain(n, seed):
    """n species of one mass, A_k <=> A_(k+1) and a few A_i + A_j <=> A_k + A_l."""
    rng = np.random.default_rng(seed)
    rx = [dict(re=[(k, 1)], pr=[(k + 1, 1)]) for k in range(n - 1)]
    for _ in range(2 * n if n >= 4 else 0):
        a, b, c, d = (int(v) for v in rng.choice(n, 4, replace=False))
        rx.append(dict(re=[(a, 1), (b, 1)], pr=[(c, 1), (d, 1)]))
    for r in rx:
        r |= dict(A=10.0 ** rng.uniform(2, 4), b=0.0, Ea=rng.uniform(0, 2e4))
    th = [(tm.const_cp_thermo(4.0, -0.2 * k, 18.0), tm.const_cp_thermo(4.0, -0.2 * k, 18.0)) for k in range(n)]
    return tm.build([0.03] * n, th, rx)


@pytest.mark.parametrize("n", [1, 2, 3, 7, 15, 16, 17, 31, 32, 40])
def test_programs_of_every_size(n):
    m = _chain(n, n)
    h, o = chem.create(m, 0), Oracle(m)
    rng = np.random.default_rng(n)
    N = 5
    T, p, dt = rng.uniform(600.0, 1800.0, N), np.full(N, 1e5), np.full(N, 1e-3)
    Y = np.ascontiguousarray(rng.dirichlet(np.ones(n), N).T)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    for method in (0, 1, 2):
        ref = o.integrate_batch(T, p, Y, dt, method=method)
        for kw in (dict(cells_per_warp=1, warps_per_cell=1), dict(warps_per_cell=2), dict(cells_per_warp=2)):
            Tg, Yg, hio = dev(T), dev(Y), torch.zeros(N, dtype=torch.float64, device="cuda")
            ns, st = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
            h.integrate(Tg, dev(p), Yg, dev(dt), hio, ns, st, method=method, **kw)
            assert np.array_equal(st.cpu().numpy(), ref["status"]), (method, kw)
            assert np.all(np.abs(Tg.cpu().numpy() - ref["T"]) <= 1e-8 * ref["T"]), (method, kw)
            assert np.all(np.abs(Yg.cpu().numpy() - ref["Y"]) <= 1e-8), (method, kw)
