"""The energy record after a step that a bounded wait ended early (PIC_ETIMEOUT, by the
test hook of the step walker): such a step is not in the record, whose next entry is its
first and reads no entry before it.  A state set afterwards is recorded from its first step."""
import numpy as np
import pytest

import paper_1308_5892_gb300 as pic
from test_gpu_ensemble import ORACLE_RUNS, _random_ensemble

pytestmark = pytest.mark.gpu


def test_a_step_that_timed_out_is_not_in_the_energy_record():
    descs, states = _random_ensemble(ORACLE_RUNS[:3], (0, 0, 0), 970)
    with pic.Context(descs, precision=pic.PIC_MIXED, sort_interval=4) as ens:
        for r, (fields, parts) in enumerate(states):
            ens.set_state(r, fields, parts)
        ens.set_flags(pic.PIC_FLAG_INJECT_STALL)
        with pytest.raises(pic.PicError) as e:
            ens.step(1)
        assert e.value.status == pic.PIC_ETIMEOUT
        ens.set_flags(0)
        for r, (fields, parts) in enumerate(states):
            assert len(ens.energy_history(r)) == 0
            ens.set_state(r, fields, parts)
        ens.step(3)
        for r in range(len(descs)):
            h = ens.energy_history(r)
            assert h.shape == (3, 4) and np.isfinite(h).all() and (h[:, 0] > 0).all()
