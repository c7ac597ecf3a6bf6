"""The mixed schedule from many start blocks: none may lose the bands' linear independence.

The free-electron cell (degenerate shells, whose pencils become nearly decoupled as they converge) and a small
cell with projectors from 200 starts, the 120^3 Gamma cell (1024 + 128 bands, whose last block has residuals of
six orders of magnitude) from a few.
"""
import numpy as np
import pytest

import synth
from tests._helpers import ensure_built, make_solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _starts(npw, M, seeds):
    import torch
    for seed in seeds:
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        x = torch.randn(2, M, npw, dtype=torch.float64, device="cuda", generator=g)
        yield seed, torch.complex(x[0], x[1])


@pytest.mark.parametrize("cell", ["free", "projectors"])
def test_small_cells(cell):
    if cell == "free":
        w = synth.tiny_workload(a=6.0, N=12, natoms=1, kb=False)
        w._vloc = np.zeros((12, 12, 12))
        kw = {}
    else:
        w = synth.tiny_workload(a=10.0, N=24, natoms=3, kb=True, ecut=0.5 * (2 * np.pi / 10.0 * 7.2) ** 2)
        kw = dict(nbuf=8)
    first = None
    with make_solver(w, block_size=8, nline=4, max_sweeps=60, precision="mixed", tol=1e-8, **kw) as s:
        for seed, X in _starts(s.npw(0), 16, range(200)):
            res = s.solve([X])                  # raises where a solve breaks down
            assert res.status == 0, (seed, res.stats)
            first = res.eig[0] if first is None else first
            assert np.abs(res.eig[0] - first).max() < 1e-9, seed


def test_gamma120():
    w = synth.make_workload("gamma120")
    first = None
    with make_solver(w, block_size=128, nline=4, max_sweeps=30, precision="mixed", tol=1e-8, nbuf=128) as s:
        for seed, X in _starts(s.npw(0), 1024, range(1, 4)):
            res = s.solve([X])
            assert res.status == 0, (seed, res.stats)
            first = res.eig[0] if first is None else first
            assert np.abs(res.eig[0] - first).max() < 1e-9, seed
