"""The loader's quick inverses over the range of temperatures: below theta = 8e-5 the
marginal's is not used, above it is with about one part in 10^5 of the mixed path's
particles done again.  FP64 momenta agree with the oracle to the accuracy of the two
tables (as in the loader's parity test), and the mixed path's are their FP32
roundings: the two differ by 1e-14 where FP32 has 6e-8, so among 10^5 values none or,
at odds of one in a hundred, one falls on the other side."""
import numpy as np
import pytest

from oracle import mj
import paper_1308_5892_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta,beta", [(2e-5, 0.0), (7e-5, 0.6), (1e-4, 0.6), (0.01, 0.0), (0.3, 0.99), (30.0, 0.3),
                                        (1e4, 0.0)])
def test_quick_inverses_match_oracle_and_round_alike(theta, beta):
    ppc, nx, ny = 24, 45, 33
    n = ppc * nx * ny
    d = pic.run_desc(2, nx, ny, 1, 2.0, 16.0, 0.5, [(-1.0, 1.0, n)])
    got = []
    for precision in (pic.PIC_FP64, pic.PIC_MIXED):
        with pic.Context([d], precision=precision) as ctx:
            ctx.load_maxwell_juttner(0, 0, ppc, theta, (0.0, 0.0, beta), seed=77)
            got.append(ctx.get_state(0)[1][0][3:])
    _, ref = mj.load(77, 0, n, theta, (0.0, 0.0, beta), 2, nx, ny, 1)
    assert got[0].shape[1] == n
    assert np.abs(got[0] - ref).max() <= 1e-9 * max(1.0, np.abs(ref).max())
    assert (got[0].astype(np.float32) != got[1].astype(np.float32)).sum() <= 1
