"""Rounds of simple reactions (A + B <=> C + D, four species, no third body) and of all others, against the oracle.

A round of lanes whose reactions are all simple takes a short form of the rate of progress and of its
derivatives; any other reaction in it sends the whole round to the general form.  Counts at the edges of a
round (16, 32 and 64 lanes) with and without other kinds: a species repeated on one side, the same species on
both sides, irreversible, three reactants, two products less, third-body and fall-off reactions.
Tolerances: 1e-12 of the gross size of the terms for the source term and the Jacobian, 1e-8 for a short
integration with each kind of lane group.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.oracle import Oracle  # noqa: E402
from paper_2311_14941_gb300 import chem  # noqa: E402
from tests import tinymech as tm  # noqa: E402

N_SP = 7
OTHERS = [dict(re=[(0, 2)], pr=[(1, 1), (2, 1)]), dict(re=[(0, 1), (1, 1)], pr=[(0, 1), (2, 1)]),
          dict(re=[(2, 1), (3, 1)], pr=[(4, 1), (5, 1)], rev=0), dict(re=[(0, 1), (1, 2)], pr=[(3, 1), (6, 1)]),
          dict(re=[(4, 1), (5, 1)], pr=[(6, 1)]), dict(re=[(3, 1), (4, 1)], pr=[(5, 3)]),
          dict(re=[(0, 1), (5, 1)], pr=[(2, 1)], type=1, eff={1: 3.0, 4: 0.5}),
          dict(re=[(1, 1), (3, 1)], pr=[(4, 1)], type=2, eff={0: 2.0, 6: 0.0}, troe=[0.6, 100.0, 2000.0, 3000.0],
               low=[2.0, -0.5, 1.0e4]),
          dict(re=[(6, 2)], pr=[(0, 1)], type=2, eff={2: 5.0}, troe=[0.4, 300.0, 1500.0, 0.0], low=[1.5, 0.0, 5.0e3])]


def _mechanism(n_simple, n_other, seed):
    rng = np.random.default_rng(seed)
    rx = []
    for _ in range(n_simple):
        a, b, c, d = rng.choice(N_SP, 4, replace=False)
        rx.append(dict(re=[(int(a), 1), (int(b), 1)], pr=[(int(c), 1), (int(d), 1)]))
    for i in range(n_other):
        rx.insert(int(rng.integers(0, len(rx) + 1)), dict(OTHERS[i % len(OTHERS)]))
    for r in rx:
        r |= dict(A=10.0 ** rng.uniform(0, 3), b=rng.uniform(-1, 1), Ea=rng.uniform(0, 4e4))
    th = [(tm.const_cp_thermo(3.0 + 0.3 * k, -2.0 * k, 18.0 + k), tm.const_cp_thermo(3.0 + 0.3 * k, -2.0 * k, 18.0 + k))
          for k in range(N_SP)]
    return tm.build([0.02 + 0.003 * k for k in range(N_SP)], th, rx)


def _states(N, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(400.0, 2200.0, N), rng.uniform(5e4, 5e5, N),
            np.ascontiguousarray(rng.dirichlet(np.ones(N_SP), N).T))


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("n_simple,n_other", [(1, 0), (15, 1), (16, 0), (31, 2), (32, 0), (33, 9), (63, 1), (64, 0), (65, 9),
                                              (0, 9), (97, 3)])
def test_rounds_of_reactions(n_simple, n_other):
    m = _mechanism(n_simple, n_other, 100 * n_simple + n_other)
    h, o = chem.create(m, 0), Oracle(m)
    N = 9
    T, p, Y = _states(N, n_simple)
    f8 = lambda *s: torch.empty(*s, dtype=torch.float64, device="cuda")
    dT, dY, S, u, v = f8(N), f8(N_SP, N), f8(h.info["nnz_S"], N), f8(h.m, N), f8(h.m, N)
    h.rates(_dev(T), _dev(p), _dev(Y), dT, dY)
    h.jacobian(_dev(T), _dev(p), _dev(Y), S, u, v)
    torch.cuda.synchronize()
    rp, ci = h.jacobian_pattern()
    for c in range(N):
        r = o.rhs(T[c], p[c], Y[:, c], want_gross=True)
        f = np.r_[dT[c].item(), dY[:, c].cpu().numpy()]
        assert np.all(np.abs(f - r["f"]) <= 1e-12 * (np.abs(r["f"]) + r["gross"]) + 1e-300)
        Jg = np.outer(u[:, c].cpu().numpy(), v[:, c].cpu().numpy())
        Sc = S[:, c].cpu().numpy()
        for row in range(h.m):
            Jg[row, ci[rp[row]:rp[row + 1]]] += Sc[rp[row]:rp[row + 1]]
        J, G = o.jacobian(T[c], p[c], Y[:, c], want_gross=True)
        assert np.all(np.abs(Jg - J) <= 1e-12 * (np.abs(J) + G) + 1e-300)
    dt = np.full(N, 1e-5)
    ref = o.integrate_batch(T, p, Y, dt)
    for kw in (dict(cells_per_warp=1, warps_per_cell=1), dict(warps_per_cell=2), dict(cells_per_warp=2)):
        Tg, Yg, hio = _dev(T), _dev(Y), torch.zeros(N, dtype=torch.float64, device="cuda")
        ns, st = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
        h.integrate(Tg, _dev(p), Yg, _dev(dt), hio, ns, st, **kw)
        # (the random sets that do not conserve mass blow up: the oracle's cells end the same way)
        assert np.array_equal(st.cpu().numpy(), ref["status"]), kw
        ok = ref["status"] == 0
        assert np.all(np.abs(Tg.cpu().numpy() - ref["T"])[ok] <= 1e-8 * ref["T"][ok]), kw
        assert np.all(np.abs(Yg.cpu().numpy() - ref["Y"])[:, ok] <= 1e-8), kw
