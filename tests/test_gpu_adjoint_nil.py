"""Reactions that change nothing (the same species on both sides): whatever their rate of progress, infinite and NaN
included, the state's adjoint does not see them.  With no other reaction the state stays as it is, and the gradients with
respect to the initial state are those given for the final one, bit for bit (tolerance 0); at 1e-3 K exp(g) overflows and
the rate is NaN.  Beside other reactions the gradients are those of the mechanism without the idle ones, to the rounding
that their place among the others leaves (1e-12 of the largest).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_14941_gb300 import chem, synth  # noqa: E402
from tests import tinymech as tm  # noqa: E402
from tests.test_gpu_adjoint import _adjoint  # noqa: E402

N_SP = 5
IDLE = [dict(re=[(0, 1)], pr=[(0, 1)], A=3.0, b=0.5, Ea=1e4), dict(re=[(1, 1), (2, 1)], pr=[(2, 1), (1, 1)], A=2e2, b=0.0, Ea=5e3),
        dict(re=[(3, 2)], pr=[(3, 2)], A=5.0, b=0.0, Ea=2e4, type=1, eff={4: 3.0})]
OTHERS = [dict(re=[(0, 1), (1, 1)], pr=[(2, 1), (3, 1)], A=2e3, b=0.0, Ea=1e4), dict(re=[(2, 1)], pr=[(4, 1)], A=1e3, b=0.0, Ea=2e4)]


def _run(reactions, T, n_cells=3):
    th = [(tm.const_cp_thermo(4.0, -0.2 * k, 18.0), tm.const_cp_thermo(4.0 + 0.1 * k, -0.3 * k, 17.0)) for k in range(N_SP)]
    h = chem.create(tm.build([0.03] * N_SP, th, reactions), 0)
    rng = np.random.default_rng(4)
    F = synth.Field(np.full(n_cells, T), np.full(n_cells, 1e5), np.ascontiguousarray(rng.dirichlet(np.ones(N_SP), n_cells).T),
                    np.full(n_cells, 1e-4), np.zeros(n_cells, dtype=np.int32))
    gT, gY = rng.standard_normal(n_cells) * 1e-3, rng.standard_normal((N_SP, n_cells))
    return F, gT, gY, _adjoint(h, F, gT, gY, torch.device("cuda:0"))


@pytest.mark.parametrize("T", [1e-3, 300.0, 1500.0])
def test_idle_reactions_leave_the_adjoint_alone(T):
    F, gT, gY, g = _run(IDLE, T)
    assert np.all(g["status"] == 0) and np.array_equal(g["T"], F.T) and np.array_equal(g["Y"], F.Y)
    assert np.array_equal(g["gT0"], gT) and np.array_equal(g["gY0"], gY)


def test_idle_reactions_beside_others():
    a, b = _run(IDLE + OTHERS, 1500.0)[3], _run(OTHERS, 1500.0)[3]
    assert np.all(a["status"] == 0) and np.all(b["status"] == 0)
    for k in ("gT0", "gY0"):
        assert np.max(np.abs(a[k] - b[k])) <= 1e-12 * np.max(np.abs(b[k]))
    k, n = len(IDLE), len(OTHERS)
    R = k + n
    for at, bt in ((slice(k, R), slice(0, n)), (slice(R + k, 2 * R), slice(n, 2 * n))):
        assert np.max(np.abs(a["gc"][at] - b["gc"][bt])) <= 1e-12 * np.max(np.abs(b["gc"][bt]))
