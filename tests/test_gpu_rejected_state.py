"""A rejected FP64 upload leaves its run in the context, and pic_step advances every
run: the positions that failed must index inside the grid, and the other runs go on
as without it.  Over the plain, the sorted (grids of about 10^6 cells) and the direct
path (fewer particles than a fifth of the cells), in 2D and 3D, periodic and between
walls.  Bound: the order of the current sums, a few 1e-16 of each array's largest value
per step."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
from test_gpu_parity import _make

pytestmark = pytest.mark.gpu

BAD = [np.nan, np.inf, -np.inf, -1.0, -1e-300, -3e9, 1e300, 2.0 ** 21, 2.0 ** 40 + 0.5]


@pytest.mark.parametrize("ndim,shape,ppc,bc", [(2, (16, 12, 1), 4, 0), (3, (7, 9, 8), 2, 0), (2, (21, 12, 1), 4, 1),
                                               (2, (1100, 900, 1), 0.01, 0), (3, (91, 100, 88), 0.01, 1),
                                               (2, (1100, 900, 1), 0.15, 0), (3, (91, 100, 88), 0.15, 1)])
def test_other_runs_go_on_after_a_rejected_fp64_state(ndim, shape, ppc, bc):
    desc, fields, parts, _ = _make(ndim, shape, ppc, seed=61 + ndim, spread=0.5, amp=0.01, colocate=False, bc=(bc, 0, 0))
    if bc:   # what vanishes on the wall
        fields[1][..., 0] = fields[2][..., 0] = fields[3][..., 0] = 0.0
    bad = [p.copy() for p in parts]
    for k, v in enumerate(BAD):
        bad[k % 2][k % ndim, 3 * k] = v
    with pic.Context([desc, desc], precision=pic.PIC_FP64) as two, pic.Context([desc], precision=pic.PIC_FP64) as one:
        two.set_state(1, fields, parts)
        one.set_state(0, fields, parts)
        with pytest.raises(pic.PicError) as e:
            two.set_state(0, fields, bad)
        assert e.value.status in (pic.PIC_EINVAL, pic.PIC_ENUMERIC)
        for n in (1, 2):
            two.step(n)
            one.step(n)
        f2, p2, _ = two.get_state(1)
        f1, p1, _ = one.get_state(0)
        # the rejected run itself: every particle in the domain
        for p in two.get_state(0)[1]:
            for a in range(ndim):
                assert p[a].min() >= 0.0 and p[a].max() <= shape[a]
        # and a good state is taken again
        two.set_state(0, fields, parts)
        two.step(1)
    assert np.abs(f2 - f1).max() <= 1e-13 * np.abs(f1).max()
    for a, b in zip(p2, p1):
        assert np.abs(a - b).max() <= 1e-13 * max(shape)
