"""The internal order formed on the device: a context in lattice-line order
equals, bit for bit, one in the caller's order whose caller sorted the
particles by the order's definition (numpy), at line lengths on either side of
the block sort's shared-memory limit and with unequal volumes; and the
order found again (TLSPH_FLAG_AUTO_ORDER) in one creation."""
import dataclasses

import numpy as np
import pytest

from paper_1901_07374_gb300 import specimen as S
from paper_1901_07374_gb300 import tlsph

pytestmark = pytest.mark.gpu


def _line_order(X, vol):
    lo, ext = X.min(0), X.max(0) - X.min(0)
    L = int(np.argmax(ext))
    a, b = (L + 1) % 3, (L + 2) % 3
    d = np.cbrt(np.partition(vol, len(vol) // 2)[len(vol) // 2])
    inv = 1.0 / d
    ka = np.floor((X[:, a] - lo[a]) * inv + 0.5)
    kb = np.floor((X[:, b] - lo[b]) * inv + 0.5)
    t = np.floor((X[:, L] - lo[L]) * (4294967295.0 / ext[L]))
    return np.lexsort((np.arange(len(X)), t, kb, ka))


def _permuted(w, perm):
    sp = w.specimen
    return dataclasses.replace(w, specimen=dataclasses.replace(
        sp, X=np.ascontiguousarray(sp.X[perm]), vol=sp.vol[perm].copy(), mat_id=sp.mat_id[perm].copy(),
        bc_mask=sp.bc_mask[perm].copy(), bc_vel=np.ascontiguousarray(sp.bc_vel[perm]), f0=sp.f0[perm].copy()))


CASES = [("bar", 7, 9, 33, False), ("long", 3, 3, 2047, False), ("past_shared", 3, 3, 2300, False),
         ("shuffled", 12, 11, 40, True), ("volumes", 8, 8, 20, True)]


@pytest.mark.parametrize("name,nx,ny,nz,shuffle", CASES)
def test_line_order_equals_its_definition(name, nx, ny, nz, shuffle):
    w = S.tensile_bar_cl(nx, ny, nz, v_grip=1.0)
    rng = np.random.default_rng(5)
    if shuffle:
        w = _permuted(w, rng.permutation(w.specimen.N))
    if name == "volumes":
        w.specimen.vol = w.specimen.vol * (1.0 + 0.02 * rng.random(w.specimen.N))
    perm = _line_order(w.specimen.X, w.specimen.vol)
    a = tlsph.Simulation.from_workload(w, precision="mixed", line_order=True)
    b = tlsph.Simulation.from_workload(_permuted(w, perm), precision="mixed", line_order=False)
    assert a.neighbor_layout() == b.neighbor_layout()
    for s in (a, b):
        s.step(5)
        s.sync()
    for k, v in b.state().items():
        assert np.array_equal(a.get(k)[perm], v), k
        assert np.array_equal(a.get_device(k).cpu().numpy()[perm], v), k


def test_order_found_again_in_one_creation():
    w = S.taylor_impact(6000)
    auto, line = (tlsph.Simulation.from_workload(w, precision="mixed", line_order=o) for o in (None, True))
    own = tlsph.Simulation.from_workload(w, precision="mixed", line_order=False)
    assert own.neighbor_layout()["aligned_slices"] < 0.9 * own.neighbor_layout()["slices"]
    assert auto.neighbor_layout() == line.neighbor_layout() != own.neighbor_layout()
    # a body whose lines align no more than the caller's order keeps the caller's
    shuffled = _permuted(w, np.random.default_rng(1).permutation(w.specimen.N))
    shuffled.specimen.vol = shuffled.specimen.vol * 1e-3        # lattice spacing far from the positions': no lines
    auto2, own2 = (tlsph.Simulation.from_workload(shuffled, precision="mixed", line_order=o) for o in (None, False))
    for s in (auto, line, auto2, own2):
        s.step(4)
        s.sync()
    for k, v in line.state().items():
        assert np.array_equal(auto.get(k), v), k
    if auto2.neighbor_layout() == own2.neighbor_layout():
        for k, v in own2.state().items():
            assert np.array_equal(auto2.get(k), v), k
