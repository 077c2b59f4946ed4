"""The sort counts and ranks the particles of an old tile over the cells of its box in
shared memory; untiled sources, tiles whose box does not fit and particles beyond the box
take the general form.  Neither the tile nor the form enters the result (currents are exact
sums, and every particle is advanced by the same arithmetic), so fields and particles are
bitwise equal over tiles: a box that does not fit, sides that are no powers of two, one
cell wide, and species on both sides of the size that decides about shared launches; with
particles fast enough to leave the box between sorts."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5003, 61000])
@pytest.mark.parametrize("interval", [1, 7])
def test_tiles_and_sort_forms_equal_bitwise(n, interval):
    nx, ny = 83, 71
    rng = np.random.default_rng(n + interval)
    f = rng.normal(0.0, 0.05, (6, 1, ny, nx))
    parts = [np.concatenate([synth.positions(rng, 2, nx, ny, 1, m), synth.momenta(rng, m, 2.0)]) for m in (n, n // 3 + 1)]
    desc = pic.run_desc(2, nx, ny, 1, 4.0, 16.0, 0.5, [(-1.0, 1.0, n), (1.0, 4.0, n // 3 + 1)])
    ref = None
    for tile in ((16, 16, 1), (64, 32, 1), (13, 7, 1), (32, 16, 1), (1, 40, 1)):
        with pic.Context([desc], tile=tile, sort_interval=interval) as ctx:
            ctx.set_state(0, f, parts)
            ctx.step(2 * interval + 3)
            got = ctx.get_state(0)
        if ref is None:
            ref = got
        np.testing.assert_array_equal(got[0], ref[0])
        for a, b in zip(got[1], ref[1]):
            np.testing.assert_array_equal(a, b)
