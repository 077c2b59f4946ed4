"""FP64 runs with fewer particles than a fifth of the cells gather and deposit at the
particle, others by node averages and moments.  Both sides of the line against the oracle,
and a run that crosses it by a load, which must not find the current of the other form in
its ghost cells: against a run in which nothing but the load's state has been."""
import numpy as np
import pytest

import oracle
import paper_1308_5892_gb300 as pic
from test_gpu_parity import _compare, _make, _oracle_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,shape,bc", [(2, (40, 30, 1), 0), (2, (29, 40, 1), 1), (3, (12, 10, 10), 0), (3, (11, 12, 10), 1)])
@pytest.mark.parametrize("n", ["few", "below", "at"])   # per species; the line is at cells / 10 of each of two
def test_both_sides_of_the_line_match_oracle(ndim, shape, bc, n):
    desc, fields, parts, arr = _make(ndim, shape, 1, seed=430 + ndim, spread=2.0, amp=0.02, colocate=False, bc=(bc, 0, 0))
    if bc:   # what vanishes on the wall
        fields[1][..., 0] = fields[2][..., 0] = fields[3][..., 0] = 0.0
    cells = int(np.prod(shape))
    m = {"few": 3, "below": (cells - 1) // 10, "at": cells // 10 + 1}[n]
    parts = [np.ascontiguousarray(p[:, :m]) for p in parts]
    for s, p in zip(arr["species"], parts):
        s["pos"], s["u"] = p[:3], p[3:]
    with pic.Context([desc], precision=pic.PIC_FP64) as ctx:
        ctx.set_state(0, fields, parts)
        st = _oracle_state(desc, fields, parts, arr)
        for nsteps in (1, 4):
            ctx.step(nsteps)
            oracle.step(st, nsteps)
            f, p, _ = ctx.get_state(0)
            _compare(desc, f, p, st, 1e-12, 1e-12 * max(shape), 1e-12)


@pytest.mark.parametrize("ndim,shape", [(2, (40, 30, 1)), (3, (12, 10, 10)), (2, (1100, 900, 1))])
@pytest.mark.parametrize("order", [(0.02, 2.0), (2.0, 0.02), (0.02, 2.0, 0.02)])
def test_a_run_that_crosses_the_line_by_a_load(ndim, shape, order):
    cap = int(2 * np.prod(shape))
    desc = pic.run_desc(ndim, *shape, 2.0, 4.0, 0.5, [(-1.0, 1.0, cap), (1.0, 1.0, cap)])
    with pic.Context([desc], precision=pic.PIC_FP64) as a, pic.Context([desc], precision=pic.PIC_FP64) as b:
        f = np.zeros((6, shape[2], shape[1], shape[0]))
        none = [np.zeros((6, 0))] * 2
        a.set_state(0, f, none)
        for k, ppc in enumerate(order):
            b.set_state(0, a.get_state(0)[0], none)   # the same fields, zero current
            for ctx in (a, b):
                for s in range(2):
                    ctx.load_maxwell_juttner(0, s, ppc, 0.5, seed=10 * k + s)
                ctx.step(3)
            fa, pa, _ = a.get_state(0)
            fb, pb, _ = b.get_state(0)
            # 3 steps of sums in another order, each a few 1e-16 of the largest value
            assert np.abs(fa - fb).max() <= 1e-13 * np.abs(fa).max()
            for x, y in zip(pa, pb):
                d = np.abs(x - y)
                for q, L in zip(range(ndim), shape):
                    d[q] = np.minimum(d[q], L - d[q])
                assert d.max() <= 1e-13 * max(shape)
