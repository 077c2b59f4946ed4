"""The drift components that pic_mj_sample_marginal returns (and times) are those that the
loader draws from the same uniforms: along beta, without fields, a loaded momentum is the
drift component itself, bit for bit in the FP64 path and rounded to FP32 in the mixed path."""
import numpy as np
import pytest

from oracle import mj
import paper_1308_5892_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta,beta", [(2e-5, 0.3), (1e-3, 0.6), (0.1, 0.05), (1.0, 0.6), (10.0, 0.9), (300.0, 0.99)])
def test_exact_sampler_returns_what_the_loader_draws(theta, beta):
    nx, ny, ppc, seed = 64, 50, 31, 12
    n = nx * ny * ppc
    w = mj.uniforms(seed, 0, np.arange(n))[3]
    d = pic.run_desc(2, nx, ny, 1, 2.0, 16.0, 0.5, [(-1.0, 1.0, n)])
    for precision, kind in ((pic.PIC_FP64, np.float64), (pic.PIC_MIXED, np.float32)):
        with pic.Context([d], precision=precision) as ctx:
            y, ms = ctx.mj_sample_marginal(theta, beta, w, method=pic.PIC_MJ_EXACT)
            ctx.load_maxwell_juttner(0, 0, ppc, theta, (0.0, 0.0, beta), seed=seed)
            uz = ctx.get_state(0)[1][0][5]
        assert ms > 0
        differ = (y.astype(kind) != uz.astype(kind)).sum()
        # (the mixed path draws once more in full where FP32 could round otherwise: one in 10^5, and of
        # those few have another rounding)
        assert differ <= (0 if kind is np.float64 else 2), (precision, differ)
