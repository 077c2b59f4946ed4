"""Any number of particles in one cell, all moving alike: the push sums a lane's fluxes of
a cell in 32-bit registers, at most 32 particles at a time.  All particles of a species
share one state and the fields are zero, so one step's current is that of one particle
times their number: the oracle takes one particle per species with the charge density
that many times smaller.  The mixed path rounds the momenta to FP32 (6e-8) and each flux
to 2^-27 (2e-8 of these), far below the bound."""
import numpy as np
import pytest

import oracle
import paper_1308_5892_gb300 as pic

pytestmark = pytest.mark.gpu

N_X, RHO, DT = 4.0, 64.0, 0.5


@pytest.mark.parametrize("ndim,shape,n,flags,runs", [
    (2, (16, 12, 1), 50000, pic.PIC_FLAG_PHASE_LAUNCHES, 2), (2, (128, 128, 1), 50000, 0, 2), (2, (16, 12, 1), 50000, 0, 1),
    (2, (40, 24, 1), 700000, 0, 5), (2, (32, 32, 1), 9000000, 0, 1), (3, (9, 8, 10), 120000, pic.PIC_FLAG_PHASE_LAUNCHES, 2),
    (3, (48, 48, 48), 150000, 0, 2), (3, (12, 12, 12), 9000000, 0, 1)])
def test_coherent_particles_of_one_cell(ndim, shape, n, flags, runs):
    states = [np.array([5.25, 5.0625, 5.125 if ndim == 3 else 0.0, 3.0, 1.0, 0.5]),
              np.array([5.75, 5.9375, 5.875 if ndim == 3 else 0.0, -3.0, -1.0, -0.5])]
    nx, ny, nz = shape
    st = oracle.State.empty(ndim, nx, ny, nz, DT, N_X, RHO / n)
    for x, q in zip(states, (1.0, -1.0)):
        st.species.append(oracle.Species(np.ascontiguousarray(x[:3, None]), np.ascontiguousarray(x[3:, None]), q, 1.0))
    desc = pic.run_desc(ndim, nx, ny, nz, N_X, RHO, DT, [(1.0, 1.0, n), (-1.0, 1.0, n)])
    fields = np.zeros((6, nz, ny, nx))
    with pic.Context([desc] * runs, flags=flags) as ctx:
        for r in range(runs):
            ctx.set_state(r, fields, [np.repeat(x[:, None], n, axis=1) for x in states])
        ctx.step(1)
        oracle.step(st)
        for r in range(runs):
            got, _, _ = ctx.get_state(r, fields_only=True)
            for c in range(3):
                assert np.abs(got[c] - st.e[c]).max() <= 1e-6 * np.abs(st.e).max(), (r, c)
