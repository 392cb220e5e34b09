"""The FP64 step's row sums at the sizes where their form changes: particle
counts on either side of the lane rules and of a block's rows, with damaged
and undamaged neighbours and two materials, against the oracle (TOL_FP64: the
sums over j are regrouped, nothing else) -- and with the pair table
(library-owned memory) against without it (caller arena), bit for bit."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1901_07374_gb300 import specimen as S
from paper_1901_07374_gb300 import tlsph
from parity import compare_state

pytestmark = pytest.mark.gpu


def _workload(n, hg):
    base = S.tensile_bar_cl()
    nx = 16 if n > 500 else 4
    X, _ = S.lattice_box(nx, nx, -(-n // (nx * nx)), base.specimen.spacing)
    rng = np.random.default_rng(n)
    X = (X + rng.uniform(-0.01, 0.01, X.shape) * base.specimen.spacing)[:n]
    d = base.specimen.spacing
    sp = S.Specimen("rows", X, np.full(n, d ** 3), (np.arange(n) % 3 == 0).astype(np.int32), np.zeros(n, np.uint8),
                    rng.normal(size=(n, 3)) * 2.0, np.zeros(n), d)
    stiff = dict(base.materials[0], E=200e9)
    return dataclasses.replace(base, specimen=sp, materials=[base.materials[0], stiff], hg_alpha=hg)


@pytest.mark.parametrize("hg", [10.0, 0.0])
@pytest.mark.parametrize("n", [31, 33, 4095, 4099, 8191, 8195])
def test_rows_with_and_without_table(n, hg):
    import torch
    w = _workload(n, hg)
    rng = np.random.default_rng(3)
    dinit = np.where(rng.random(n) < 0.3, 1.0 + 0.09 * rng.random(n), 0.0)
    D = np.where(dinit >= 1.0, 10.0 * (dinit - 1.0), 0.0)
    a = tlsph.Simulation.from_workload(w)
    nbytes = tlsph.workspace_bytes(a.cfg, n, a.nnz)
    arena = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    b = tlsph.Simulation.from_workload(w, arena=arena, nnz_cap=a.nnz)
    o = oracle.Simulation.from_workload(w, neighbors_csr=(a.get("NBR_ROWPTR"), a.get("NBR_COL")))
    o["dinit"][:], o["D"][:] = dinit, D
    for s in (a, b):
        s.set("DINIT", dinit)
        s.set("DAMAGE", D)
        s.step(3)
    o.step(3)
    compare_state(a.state(), o.state(), w)
    for k, v in a.state().items():
        assert np.array_equal(b.get(k), v), k
