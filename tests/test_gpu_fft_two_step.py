"""Local-potential passes in two steps per line (N = R1 R2), every grid edge that has its own kernels,
against the oracle's H: the half box (default cutoff: at most N / 2 + 1 planes and rows) and a wider
sphere, general and Gamma k-points, and band counts that leave a short last batch.

Tolerances: those of the other H tests, relative to max |Hx|.
"""
import numpy as np
import pytest

import synth
from tests._helpers import ensure_built, make_solver, oracle_for

pytestmark = pytest.mark.gpu
EDGES = [24, 36, 40, 48, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 160]
TOL = {"c128": 1e-12, "df32": 5e-12, "c64": 5e-6}


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _check(w, nb, prec):
    import torch
    with make_solver(w, block_size=4) as s:
        H = oracle_for(w, s)
        rng = np.random.default_rng(w.N + nb)
        x = rng.standard_normal((nb, s.npw())) + 1j * rng.standard_normal((nb, s.npw()))
        if prec == "c64":
            x = x.astype(np.complex64)
        y = s.apply_H(0, torch.tensor(x, device="cuda"), df32=prec == "df32").cpu().numpy()
        want = H.apply(x.astype(np.complex128).T).T
        assert np.abs(y - want).max() < TOL[prec] * np.abs(want).max()


@pytest.mark.parametrize("prec", ["df32", "c128", "c64"])
@pytest.mark.parametrize("N", EDGES)
def test_half_box(N, prec):
    _check(synth.tiny_workload(a=0.3 * N, N=N, natoms=2, kb=False, kpt=(0.25, -0.125, 0.375) if N % 3 else (0, 0, 0)), 3, prec)


@pytest.mark.parametrize("prec", ["df32", "c128", "c64"])
@pytest.mark.parametrize("N", [24, 36, 40, 54, 60])
def test_wider_sphere(N, prec):
    a = 0.3 * N
    _check(synth.tiny_workload(a=a, N=N, natoms=2, kb=False, kpt=(0.25, 0.0, -0.5), ecut=2.5 * synth.default_ecut(a, N)),
           2, prec)


@pytest.mark.parametrize("prec", ["df32", "c128"])
def test_short_last_batch(prec):
    _check(synth.tiny_workload(a=21.0, N=96, natoms=1, kb=False, kpt=(0.25, 0.25, 0.25)), 41, prec)
