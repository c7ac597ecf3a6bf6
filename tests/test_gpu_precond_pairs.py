"""The preconditioner of the mixed schedule in double-FP32: bands whose kinetic energy is ordinary, far below every
other plane wave's (weak potentials) and nearly none (a free electron's lowest band at, or 1e-20 from, Gamma: the
Teter ratio is then so small for every other plane wave that the last digits of the residual stay).

Tolerance: the eigenvalue checks of the other solves, 1e-9 Ha.
"""
import numpy as np
import pytest

import synth
from tests._helpers import ensure_built, make_solver, oracle_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("kx", [0.0, 1e-20, 0.25])
@pytest.mark.parametrize("strength", [0.0, 1e-9, 1e-3, 1.0])
def test_lowest_band(strength, kx):
    import torch
    w = synth.tiny_workload(a=6.0, N=12, natoms=1, kb=False, kpt=(kx, 0.0, 0.0))
    w._vloc = w.vloc() * strength
    with make_solver(w, block_size=1, nline=4, max_sweeps=40, tol=1e-8, precision="mixed") as s:
        H = oracle_for(w, s)
        X = torch.tensor(synth.start_vectors(3, s.npw(0), 1).T.copy(), device="cuda")
        r = s.solve([X])
        x = X.cpu().numpy()[0]
        want = np.linalg.eigvalsh(H.apply(np.eye(s.npw(0), dtype=complex)))[0]
        assert np.isfinite(x).all()
        assert abs(r.eig[0][0] - want) < 1e-9
