"""The FP64 sort by cell where a lane of the push walks several particles: walks of 2 and 4
(from 16 rows of 32 x 2 and 32 x 4 particles per resident warp on: 2.5 and 5 million per
species; the sizes of test_gpu_fp64_sort.py all have walks of 1), with a partial last block,
beside a species of few particles.  Against the same run without the sort's scratch, which
steps in storage order: the order of the current sums is all that differs, a few 1e-16 of
each array's largest value per step.  And at densities that sort (from a fifth of a particle
per cell on): the scratch refused in part, and a partner loaded onto a sorted species."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
from test_gpu_fp64_direct import _Allocator

pytestmark = pytest.mark.gpu

WALK2, WALK4 = 16 * 152 * 16 * 64, 16 * 152 * 16 * 128   # particles from which a lane walks 2, 4


def _steps(ctx, ndim, shape, counts, steps):
    cells = float(np.prod(shape))
    for s, n in enumerate(counts):
        ctx.load_maxwell_juttner(0, s, n / cells, 0.3, seed=21 + s)
    ctx.set_uniform_field(0, (0.01, -0.02, 0.005), (0.02, 0.01, -0.01))
    out = []
    for n in steps:
        ctx.step(n)
        out.append(ctx.get_state(0))
    return out


@pytest.mark.parametrize("ndim,shape,counts,bc", [
    (2, (1100, 900, 1), (WALK2 - 1, WALK2 + 33), 0), (2, (1000, 1001, 1), (WALK4 + 4099, 500), 1),
    (3, (96, 91, 100), (WALK2 + 2047, WALK4 + 1), 0), (3, (90, 99, 93), (WALK4 + 12345, WALK2), 1)])
def test_walks_equal_storage_order(monkeypatch, ndim, shape, counts, bc):
    desc = pic.run_desc(ndim, *shape, 2.0, 8.0, 0.5, [(-1.0, 1.0, n) for n in counts], bc=(bc, 0, 0))
    desc.species[1].q_over_e = 1.0
    alloc = _Allocator(monkeypatch)
    got = []
    for short in (0, 7):   # 7 requests for the sort's scratch
        with alloc.context([desc], short) as ctx:
            got.append(_steps(ctx, ndim, shape, counts, (1, 2, 15)))   # sorts at steps 1 and 17
    for (f, p, _), (g, q, _) in zip(*got):
        assert np.abs(f - g).max() <= 1e-12 * np.abs(f).max()
        for a, b in zip(p, q):
            d = np.abs(a - b)
            for x, L in zip(range(ndim), shape):
                d[x] = np.minimum(d[x], L - d[x])
            assert d.max() <= 1e-12 * max(shape)


def test_scratch_refused_in_part(monkeypatch):
    shape, n = (1100, 900, 1), 150000
    desc = pic.run_desc(2, *shape, 2.0, 8.0, 0.5, [(-1.0, 1.0, n), (1.0, 1.0, n)])
    alloc = _Allocator(monkeypatch)
    got = []
    for short in (0, 3, 7):
        with alloc.context([desc], short) as ctx:
            got.append(_steps(ctx, 2, shape, (n, n), (3,))[0])
    for f, p, _ in got[1:]:
        assert np.abs(f - got[0][0]).max() <= 1e-13 * np.abs(f).max()
        for a, b in zip(p, got[0][1]):
            assert np.abs(a - b).max() <= 1e-13 * max(shape)


def test_partner_of_a_sorted_species():
    n = 300000
    desc = pic.run_desc(2, 1000, 1000, 1, 2.0, 0.6, 0.5, [(-1.0, 1.0, n), (1.0, 1.0, n)])
    with pic.Context([desc], precision=pic.PIC_FP64) as ctx:
        ctx.load_maxwell_juttner(0, 0, 0.3, 0.5, seed=5)
        ctx.step(2)
        ctx.load_maxwell_juttner(0, 1, 0.3, 0.5, colocate_with=0, seed=6)
        _, p, _ = ctx.get_state(0)
        np.testing.assert_array_equal(p[0][:2], p[1][:2])
        ctx.step(2)
        q = ctx.get_particles(0, 1, np.arange(0, n, 1009))
        np.testing.assert_array_equal(q, ctx.get_state(0)[1][1][:, ::1009])
