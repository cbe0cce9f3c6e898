"""Gradients where the contracted products with the Jacobian take their less usual forms, against the oracle's
complex step (tests/test_gpu_adjoint.py's criterion, 1e-7 of the gradient's norm): many species and one reaction
(the dual-number cell does not fit the forward cell's shared memory), many reactions of few species (the
derivative slots do not fit the Jacobian's place), every kind of reaction, irreversible ones included, and round
counts at the edge of a warp.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.oracle import Oracle  # noqa: E402
from paper_2311_14941_gb300 import chem, synth  # noqa: E402
from tests import tinymech as tm  # noqa: E402
from tests.test_gpu_adjoint import _adjoint, _check_cell  # noqa: E402
from tests.test_gpu_reactions import OTHERS, _mechanism  # noqa: E402


def _one_reaction(n):
    th = [(tm.const_cp_thermo(4.0, -0.2 * k, 18.0), tm.const_cp_thermo(4.0, -0.2 * k, 18.0)) for k in range(n)]
    return tm.build([0.03] * n, th, [dict(re=[(0, 1)], pr=[(n - 1, 1)], A=3e3, b=0.0, Ea=1e4)])


def _conserving(kinds):
    """Reactions of OTHERS (by index) that keep the number of molecules, each once more reversed in role."""
    m = [dict(OTHERS[i]) | dict(A=50.0 * (i + 1), b=0.3, Ea=5e3 * (i + 1)) for i in kinds]
    th = [(tm.const_cp_thermo(3.5 + 0.2 * k, -0.5 * k, 18.0), tm.const_cp_thermo(3.5 + 0.2 * k, -0.5 * k, 18.0))
          for k in range(7)]
    return tm.build([0.02] * 7, th, m)


@pytest.mark.parametrize("name,dt", [("one reaction of 40 species", 1e-4), ("97 reactions of 7 species", 1e-7),
                                     ("32 simple", 1e-7), ("every kind", 1e-7)])
def test_gradients(name, dt):
    m = (_one_reaction(40) if "40" in name else _mechanism(97, 3, 9703) if "97" in name else
         _mechanism(32, 0, 3200) if "32" in name else _conserving([0, 1, 2, 6, 7, 8]))
    h, o = chem.create(m, 0), Oracle(m)
    rng = np.random.default_rng(7)
    N, n = 3, m.n_species
    F = synth.Field(rng.uniform(800.0, 1600.0, N), rng.uniform(5e4, 3e5, N),
                    np.ascontiguousarray(rng.dirichlet(np.ones(n), N).T), np.full(N, dt), np.zeros(N, dtype=np.int32))
    gT, gY = rng.standard_normal(N) * 1e-3, rng.standard_normal((n, N))
    g = _adjoint(h, F, gT, gY, torch.device("cuda:0"))
    assert np.all(g["status"] == 0)
    R = m.n_reactions
    js = range(R) if R <= 12 else sorted(rng.choice(R, 12, replace=False).tolist())
    params = [(0, j) for j in js] + [(1, j) for j in js] + [(2, i) for i in range(0, n + 1, 1 + n // 12)]
    for c in range(N):
        _check_cell(o, F, c, g, gT, gY, params)
