"""The FP64 path's sort by cell and what depends on its storage order, against
the FP64 oracle and by id.  Grids of about 10^6 cells are sorted (every 16
steps); the sizes give partial last blocks, walks of 1 to 4 particles per lane,
empty cells, and a small species of one block.  Bounds: the order of the current
sums and the rounding of one step (a few 1e-16 of each array's largest value) are
all that differs, so 18 steps stay within 1e-12."""
import numpy as np
import pytest

import oracle
import paper_1308_5892_gb300 as pic
from test_gpu_parity import _compare, _make, _oracle_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,shape,ppc,bc,equal_caps", [
    (2, (1100, 900, 1), 0.1, 0, True), (2, (1001, 940, 1), 0.21, 1, False), (2, (1200, 850, 1), 0.0005, 0, False),
    (3, (91, 100, 88), 0.4, 0, False), (3, (100, 83, 97), 0.1, 1, True)])
def test_sorted_fp64_steps_match_oracle(ndim, shape, ppc, bc, equal_caps):
    desc, fields, parts, arr = _make(ndim, shape, ppc, seed=300 + ndim, spread=2.0, amp=0.02, colocate=False,
                                     bc=(bc, 0, 0))
    if bc:   # what vanishes on the wall
        fields[1][..., 0] = fields[2][..., 0] = fields[3][..., 0] = 0.0
    if not equal_caps:   # arrays are copied back instead of trading places
        desc.species[1].capacity += 777
    with pic.Context([desc], precision=pic.PIC_FP64) as ctx:
        ctx.set_state(0, fields, parts)
        st = _oracle_state(desc, fields, parts, arr)
        for nsteps in (1, 17):   # sorts at steps 1 and 17
            ctx.step(nsteps)
            oracle.step(st, nsteps)
            f, p, _ = ctx.get_state(0)
            _compare(desc, f, p, st, 1e-12, 1e-12 * max(shape), 1e-12)
        n = p[0].shape[1]
        ids = np.array([0, n - 1, n // 2, 17], dtype=np.int64)
        np.testing.assert_array_equal(ctx.get_particles(0, 0, ids), p[0][:, ids])
        # the energy record of step n + 1 takes the kinetic energy of step n
        ctx.step(1)
        h = ctx.energy_history(0)
        kin = sum(np.sum(np.sqrt(1.0 + (q[3:] ** 2).sum(0)) - 1.0) * s.m_over_me for q, s in zip(p, st.species))
        p2 = ctx.get_state(0)[1]
        kin2 = sum(np.sum(np.sqrt(1.0 + (q[3:] ** 2).sum(0)) - 1.0) * s.m_over_me for q, s in zip(p2, st.species))
        assert abs(h[18, 0] - 0.5 * (kin + kin2)) <= 1e-12 * kin


def _steps(desc, fields, parts, nsteps):
    with pic.Context([desc], precision=pic.PIC_FP64) as ctx:
        ctx.set_state(0, fields, parts)
        ctx.step(nsteps)
        return ctx.get_state(0)


def test_fp64_steps_unsorted_when_the_allocator_has_no_room_for_the_scratch(monkeypatch):
    import torch
    desc, fields, parts, _ = _make(2, (1100, 900, 1), 0.05, seed=311, spread=1.0, amp=0.02, colocate=False)
    real = torch.cuda.caching_allocator_alloc
    made, limit = [], [1 << 30]

    def alloc(n, *a):
        made.append(n)
        return real(n, *a) if len(made) <= limit[0] else 0

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    f0, p0, _ = _steps(desc, fields, parts, 3)
    total = len(made)
    for short in (7, 3):   # none of the seven scratch arrays, or four of them
        made.clear()
        limit[0] = total - short
        f1, p1, _ = _steps(desc, fields, parts, 3)
        assert np.abs(f1 - f0).max() <= 1e-13 * np.abs(f0).max()
        for a, b in zip(p0, p1):
            assert np.abs(a - b).max() <= 1e-13 * np.abs(a).max()


def test_loading_a_partner_of_a_sorted_species_copies_positions_by_id():
    n, ppc = 50000, 0.05
    desc = pic.run_desc(2, 1000, 1000, 1, 2.0, 0.1, 0.5, [(-1.0, 1.0, n), (1.0, 1.0, n)])
    with pic.Context([desc], precision=pic.PIC_FP64) as ctx:
        ctx.load_maxwell_juttner(0, 0, ppc, 0.5, seed=5)
        ctx.step(2)
        ctx.load_maxwell_juttner(0, 1, ppc, 0.5, colocate_with=0, seed=6)
        _, p, _ = ctx.get_state(0)
        np.testing.assert_array_equal(p[0][:2], p[1][:2])
        assert np.abs(p[0][3:] - p[1][3:]).max() > 0.1
        ctx.step(2)
        _, p, _ = ctx.get_state(0)
        assert np.isfinite(p[1]).all() and p[1][0].min() >= 0.0 and p[1][0].max() < 1000.0
