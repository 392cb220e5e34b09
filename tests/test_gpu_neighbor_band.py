"""Neighbour search with more candidates at the cutoff than a thread's list of
undecided candidates holds: an exact lattice with the cutoff at 7 spacings,
where up to 54 neighbours of a particle lie at exactly the cutoff (excluded by
the strict predicate up to the rounding of each coordinate), and the same
lattice jittered; rows equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1901_07374_gb300 import specimen as S
from paper_1901_07374_gb300 import tlsph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jitter", [0.0, 1e-9])
def test_rows_with_many_candidates_at_the_cutoff(jitter):
    import torch
    sp = S.tensile_bar(15, 14, 15, 0.5e-3, jitter=jitter)
    w = S.Workload("band", sp, [S.aluminium_cl()], 1.75e-3, 3.5e-3, 2e-8, 10.0, 1)
    row_ptr, col = oracle.neighbors(sp.X, w.rc)
    g = tlsph.Simulation.from_workload(w)
    assert np.array_equal(g.get("NBR_ROWPTR"), row_ptr)
    assert np.array_equal(g.get("NBR_COL"), col)
    X = torch.tensor(sp.X, dtype=torch.float64, device="cuda")
    rp = torch.empty(sp.N + 1, dtype=torch.int64, device="cuda")
    c = torch.empty(len(col), dtype=torch.int32, device="cuda")
    assert tlsph.neighbors_noalloc(X, w.rc, rp, c) == len(col)
    assert np.array_equal(rp.cpu().numpy(), row_ptr) and np.array_equal(c.cpu().numpy(), col)
