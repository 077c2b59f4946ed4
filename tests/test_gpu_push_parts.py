"""The push of a single run cuts tiles into parts and lets lanes walk 1 to 32
particles, by the particle total; the ensemble of the same runs pushes whole
tiles.  Every particle is advanced by the same arithmetic and currents are exact
sums, so fields and particles are bitwise equal.  The totals lie around the
lines of the rules, with all particles in one tile, and in tiles beyond the
staged box."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
import synth

pytestmark = pytest.mark.gpu


def _arrays(ndim, shape, n, seed, dense):
    rng = np.random.default_rng(seed)
    nx, ny, nz = shape
    f = rng.normal(0.0, 0.02, (6, nz, ny, nx))
    parts = []
    for _ in range(2):
        pos = synth.positions(rng, ndim, nx, ny, nz, n)
        if dense:   # most particles in a corner of the grid
            m = n - n // 7
            for a in range(ndim):
                pos[a, :m] = rng.uniform(0.0, 3.0, m)
        parts.append(np.concatenate([pos, synth.momenta(rng, n, 0.8)]))
    return f, parts


@pytest.mark.parametrize("ndim,shape,n,dense", [
    (2, (40, 24, 1), 5, False), (2, (40, 24, 1), 256, True), (2, (64, 48, 1), 32768, False), (2, (64, 48, 1), 40001, True),
    (2, (33, 50, 1), 140000, True), (2, (33, 50, 1), 262144 + 77, True), (2, (70, 61, 1), 1100003, False),
    (2, (70, 61, 1), 4300007, False), (2, (9, 7, 1), 3000, False), (3, (12, 17, 9), 6001, False),
    (3, (24, 16, 16), 70000, True), (3, (24, 16, 16), 262144, False), (3, (5, 4, 6), 20000, False)])
def test_parts_and_walks_equal_whole_tiles_bitwise(ndim, shape, n, dense):
    f, parts = _arrays(ndim, shape, n, 17 + n, dense)
    desc = pic.run_desc(ndim, *shape, 4.0, 2.0 * max(1.0, n / np.prod(shape)), 0.5, [(-1.0, 1.0, n), (1.0, 4.0, n)])
    with pic.Context([desc]) as one, pic.Context([desc, desc], flags=pic.PIC_FLAG_PHASE_LAUNCHES) as two:
        for ctx, runs in ((one, 1), (two, 2)):
            for r in range(runs):
                ctx.set_state(r, f, parts)
            ctx.step(2 * one.tuning()["sort_interval"] + 3)
        f1, p1, _ = one.get_state(0)
        f2, p2, _ = two.get_state(1)
    np.testing.assert_array_equal(f1, f2)
    for a, b in zip(p1, p2):
        np.testing.assert_array_equal(a, b)
