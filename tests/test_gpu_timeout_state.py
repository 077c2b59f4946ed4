"""After a step that a bounded wait ended early (PIC_ETIMEOUT, by the test hook of the
step walker) the state is undefined, but every later call must stay inside its arrays:
the step's sort may have named a layout that its push never wrote.  The runs are read,
diagnosed and stepped as they are, positions lie in the domain, and a state set again
steps to bitwise the result of a fresh context."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
from test_gpu_ensemble import BALANCED_3D_RUNS, BALANCED_RUNS, BALANCED_WALL_RUNS, ORACLE_RUNS, _random_ensemble

pytestmark = pytest.mark.gpu

STALL = pic.PIC_FLAG_INJECT_STALL


def _set(ctx, states):
    for r, (fields, parts) in enumerate(states):
        ctx.set_state(r, fields, parts)


def _stalled_step(ctx, n):
    ctx.set_flags(STALL | pic.PIC_FLAG_NO_GRAPH)
    with pytest.raises(pic.PicError) as e:
        ctx.step(n)
    assert e.value.status == pic.PIC_ETIMEOUT
    ctx.set_flags(0)


@pytest.mark.parametrize("runs,wall", [(BALANCED_RUNS, 0), (ORACLE_RUNS[:3], 0), (BALANCED_WALL_RUNS, 1),
                                       (BALANCED_3D_RUNS, 0), (BALANCED_3D_RUNS[::2], 1)])
# the hook hits the first sort, a later one, none; and sorts queued behind one
@pytest.mark.parametrize("before,steps,interval", [(0, 1, 4), (0, 3, 4), (4, 1, 4), (6, 2, 4), (0, 3, 1), (2, 4, 1)])
def test_calls_after_a_timeout_stay_in_range(runs, wall, before, steps, interval):
    runs = [r[:-1] + (0,) for r in runs] if wall else runs   # (no smoothing between walls)
    descs, states = _random_ensemble(runs, (wall, 0, 0), 950)
    with pic.Context(descs, precision=pic.PIC_MIXED, sort_interval=interval) as ens:
        _set(ens, states)
        ens.step(before)
        _stalled_step(ens, steps)
        for again in range(2):
            for r, d in enumerate(descs):
                _, parts, _ = ens.get_state(r)
                ens.diagnostics(r)
                for s, p in enumerate(parts):
                    for a, n in zip(range(d.ndim), (d.nx, d.ny, d.nz)):
                        assert p[a].min() >= 0.0 and p[a].max() <= n
                    ens.get_particles(r, s, np.arange(0, p.shape[1], 7))
            if again == 0:
                try:
                    ens.step(6)
                except pic.PicError as e:   # (an undefined state may hold anything the step reports)
                    assert e.status in (pic.PIC_ESTATE, pic.PIC_ENUMERIC)
        _set(ens, states)
        ens.step(5)
        got = [ens.get_state(r) for r in range(len(descs))]
    with pic.Context(descs, precision=pic.PIC_MIXED, sort_interval=interval) as ref:
        _set(ref, states)
        ref.step(5)
        for r in range(len(descs)):
            want = ref.get_state(r)
            np.testing.assert_array_equal(got[r][0], want[0])
            for a, b in zip(got[r][1], want[1]):
                np.testing.assert_array_equal(a, b)
