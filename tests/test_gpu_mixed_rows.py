"""The mixed path's row kernels for small contexts and the wide blocks of large ones (a row dealt to 2 to 16
lanes, pass 1 with its FP64 updates in one kernel) at particle counts on
either side of each rule, on aligned and explicit slices, elastic and in
plastic flow, with and without the hourglass term: the default plan against a
thread per row (pass-1 form 2, pass-2 form 1; the sums are regrouped, 1e-5 of
a field's largest value as between any two plans), and the hand-over of the
FP64-update queue between the forms."""
import dataclasses

import numpy as np
import pytest

from paper_1901_07374_gb300 import specimen as S
from paper_1901_07374_gb300 import tlsph

pytestmark = pytest.mark.gpu

FIELDS = ("U", "V", "F", "SIGMA")
SIZES = [31, 33, 4095, 4097, 8191, 8193, 19999, 20001, 49999, 50001, 99999, 100001, 399999, 400001]


def _bar(n, hg=10.0, shuffle=False, flow=True):
    base = S.tensile_bar_cl(v_grip=10.0)
    nx = 4 if n < 500 else 16
    sp = S.tensile_bar(nx, nx, -(-n // (nx * nx)), 0.5e-3, 0.01, seed=n, v_grip=10.0)
    keep = np.arange(n)
    if shuffle:
        keep = np.random.default_rng(n).permutation(n)
    sp = dataclasses.replace(sp, X=np.ascontiguousarray(sp.X[keep]), vol=sp.vol[keep], mat_id=sp.mat_id[keep],
                             bc_mask=sp.bc_mask[keep], bc_vel=np.ascontiguousarray(sp.bc_vel[keep]), f0=sp.f0[keep])
    w = dataclasses.replace(base, specimen=sp, hg_alpha=hg)
    return w, (S.plastic_flow_state(w) if flow else {})


def _sim(w, st, plan=None):
    g = tlsph.Simulation.from_workload(w, precision="mixed", line_order=False)
    if plan:
        g.set_plan(plan)
    for k, v in st.items():
        g.set(k, v)
    return g


def _close(a, b, what):
    for k in FIELDS:
        x, y = a.get(k), b.get(k)
        assert np.max(np.abs(x - y)) <= 1e-5 * max(np.max(np.abs(y)), 1e-30), (what, k)


@pytest.mark.parametrize("n", SIZES)
def test_rows_equal_a_thread_per_row(n):
    for hg, shuffle in ((10.0, False), (0.0, True)) if n < 10000 else ((10.0, n % 3 == 0),):
        w, st = _bar(n, hg, shuffle)
        a, b = _sim(w, st), _sim(w, st, (2, 128, 1, 128))
        c = _sim(w, st, None if n >= 100000 else (5, 64, 4, 128))
        for s in (a, b, c):
            s.step(3)
            s.sync()
        _close(a, b, (n, hg, shuffle))
        for k, v in a.state().items():          # forms 4 and 5 form the same weights
            assert np.array_equal(c.get(k), v), k


@pytest.mark.parametrize("n", [2000, 49000])
def test_queue_handed_over_between_forms(n):
    """Every particle is in the FP64 return: a step with the queue, steps
    without it, a step with it again and batched steps find no stale entries.
    The run equals, bit for bit, one whose every leg starts in a fresh context
    (nothing queued) from a checkpoint of the leg before."""
    w, st = _bar(n)
    a, b = _sim(w, st), _sim(w, st)
    legs = [((2, 128, 1, 128), 1), ((4, 64, 4, 128), 1), ((2, 128, 1, 128), 2), ((4, 64, 4, 128), 3),
            ((2, 128, 4, 128), 1), ("batch", 1), ((4, 64, 4, 128), 2), ("batch", 2), ((2, 128, 1, 128), 1)]
    batch = tlsph.Batch(1)

    def leg(s, plan, steps):
        if plan == "batch":
            batch.set([s])
            batch.step(steps)
            batch.sync()
        else:
            s.set_plan(plan)
            s.step(steps)
        s.sync()

    for plan, steps in legs:
        leg(a, plan, steps)
        fresh = _sim(w, {})
        fresh.restore(b.checkpoint())
        b = fresh
        leg(b, plan, steps)
    for k, v in b.state().items():
        assert np.array_equal(a.get(k), v), k
