"""Forms of the sort and of the walker's push that test_gpu_sort_paths.py and
test_gpu_ensemble.py do not reach: 3D tiles (their boxes always fit: the push's shared
memory is the tighter limit), a launch per species (more than 2^25 particles in one), a
scan of the block sums in a launch of its own (more than 2^22 keys), and an ensemble whose
tiles the walker cuts into several parts, between walls and with a sheet.  Neither the form
nor the parts enter the result, so fields and particles are bitwise equal to another form's."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
import synth

pytestmark = pytest.mark.gpu


def _same(a, b):
    np.testing.assert_array_equal(a[0], b[0])
    for x, y in zip(a[1], b[1]):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("n", [1, 4001, 60000])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("interval", [1, 5])
def test_3d_tiles_and_sort_forms_equal_bitwise(n, bc, interval):
    nx, ny, nz = 23, 20, 17
    rng = np.random.default_rng(n + 10 * bc + interval)
    f = rng.normal(0.0, 0.05, (6, nz, ny, nx))
    parts = [np.concatenate([synth.positions(rng, 3, nx, ny, nz, m), synth.momenta(rng, m, 2.0)]) for m in (n, n // 3 + 1)]
    desc = pic.run_desc(3, nx, ny, nz, 4.0, 16.0, 0.5, [(-1.0, 1.0, n), (1.0, 4.0, n // 3 + 1)], bc=(bc, 0, 0))
    ref = None
    for tile in ((8, 8, 4), (16, 8, 4), (5, 7, 3), (4, 4, 4), (8, 10, 6)):
        with pic.Context([desc], tile=tile, sort_interval=interval) as ctx:
            ctx.set_state(0, f, parts)
            ctx.step(2 * interval + 3)
            got = ctx.get_state(0)
        if ref is None:
            ref = got
        _same(got, ref)


@pytest.mark.parametrize("shape,counts", [((512, 512, 1), ((1 << 25) + 1001, 70001)),   # a launch per species
                                          ((2111, 2043, 1), (30011, 5003))])            # a scan of the block sums
def test_large_sorts_equal_those_of_an_ensemble(shape, counts):
    cells = float(np.prod(shape))
    desc = pic.run_desc(2, *shape, 4.0, max(1.0, sum(counts) / cells), 0.5, [(-1.0, 1.0, counts[0]), (1.0, 1.0, counts[1])])
    other = pic.run_desc(2, 32, 32, 1, 4.0, 8.0, 0.5, [(-1.0, 1.0, 100), (1.0, 1.0, 100)])
    got = []
    for descs in ([desc], [desc, other]):
        with pic.Context(descs, tile=(16, 16, 1), sort_interval=2,
                         flags=pic.PIC_FLAG_PHASE_LAUNCHES if len(descs) > 1 else 0) as ctx:
            for s, n in enumerate(counts):
                ctx.load_maxwell_juttner(0, s, n / cells, 0.5, seed=40 + s)
            ctx.step(5)   # sorts of an untiled and of a tiled source
            got.append(ctx.get_state(0))
    assert got[0][1][0].shape[1] == counts[0]
    _same(*got)


@pytest.mark.parametrize("ndim,bc,sheet", [(2, 1, False), (2, 1, True), (2, 0, True), (3, 1, False), (3, 1, True)])
def test_walker_with_several_parts_per_tile(ndim, bc, sheet):
    """Runs of 5000 to 20000 particles per tile: 3 to 20 parts of 1024 (one in flight's share)."""
    shapes = [(64, 32, 1), (50, 48, 1), (40, 33, 1)] if ndim == 2 else [(16, 16, 8), (19, 10, 12), (24, 9, 8)]
    descs, ppcs = [], []
    for k, shape in enumerate(shapes):
        ppc = (10, 18, 30)[k] if ndim == 2 else (12, 20, 9)[k]
        n = int(round(ppc * np.prod(shape)))
        descs.append(pic.run_desc(ndim, *shape, 4.0, 2.0 * ppc, 0.5, [(-1.0, 1.0, n), (1.0, 1.0, n)], bc=(bc, 0, 0)))
        ppcs.append(ppc)
    got = []
    for flags in (0, pic.PIC_FLAG_PHASE_LAUNCHES):
        with pic.Context(descs, sort_interval=3, flags=flags) as ens:
            for r, (shape, ppc) in enumerate(zip(shapes, ppcs)):
                for s in range(2):
                    kw = dict(profile=pic.PIC_PROFILE_HARRIS, profile_params=(shape[0] / 12.0, shape[0] / 2.0)) if sheet else {}
                    ens.load_maxwell_juttner(r, s, ppc, 1.0, (0.3, 0.0, 0.1), seed=60 + 2 * r + s, **kw)
            ens.step(8)
            got.append([ens.get_state(r) for r in range(len(descs))])
    for a, b in zip(*got):
        _same(a, b)
