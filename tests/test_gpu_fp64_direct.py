"""The FP64 path where the allocator has no room for node averages and moment planes: the
push gathers from the fields and adds to the current itself.  Against the oracle and
against the path with them; the order of the current sums and a few roundings per step
(some 1e-16 of each array's largest value) are all that differs, so 5 steps stay within
1e-12.  Memory per cell: 6 field and 3 current planes with two ghost layers, and 3 planes
for the diagnostics, no more than the 120 B of two current buffers without ghosts."""
import numpy as np
import pytest

import oracle
import paper_1308_5892_gb300 as pic
from test_gpu_parity import _compare, _make, _oracle_state

pytestmark = pytest.mark.gpu


class _Allocator:
    """torch's caching allocator, refusing every request after the first `limit`."""

    def __init__(self, monkeypatch):
        import torch
        self.real, self.sizes, self.limit = torch.cuda.caching_allocator_alloc, [], 1 << 30
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", self)

    def __call__(self, n, *a):
        if len(self.sizes) >= self.limit:
            return 0
        self.sizes.append(n)
        return self.real(n, *a)

    def context(self, descs, short=0):
        """An FP64 context whose allocator refuses the last `short` requests a full one makes."""
        self.limit, self.sizes = 1 << 30, []
        pic.Context(descs, precision=pic.PIC_FP64).close()
        self.limit, self.sizes = len(self.sizes) - short, []
        return pic.Context(descs, precision=pic.PIC_FP64)


def _case(ndim, shape, ppc, bc, smooth, seed):
    desc, fields, parts, arr = _make(ndim, shape, ppc, seed=seed, spread=2.0, amp=0.02, colocate=False, bc=(bc, 0, 0))
    desc.smooth_passes = smooth
    if bc:   # what vanishes on the wall
        fields[1][..., 0] = fields[2][..., 0] = fields[3][..., 0] = 0.0
    return desc, fields, parts, arr


@pytest.mark.parametrize("ndim,shape,ppc,bc,smooth", [
    (2, (33, 20, 1), 4, 0, 0), (2, (21, 30, 1), 5, 1, 0), (2, (2, 3, 1), 40, 0, 0), (2, (31, 18, 1), 4, 0, 2),
    (3, (12, 10, 9), 3, 0, 0), (3, (9, 11, 10), 3, 1, 0), (3, (2, 2, 3), 30, 0, 0), (3, (10, 9, 8), 3, 0, 1)])
@pytest.mark.parametrize("short", [1, 2])   # the moment planes alone are refused, or both
def test_direct_fp64_steps_match_oracle(monkeypatch, ndim, shape, ppc, bc, smooth, short):
    desc, fields, parts, arr = _case(ndim, shape, ppc, bc, smooth, 400 + ndim)
    with _Allocator(monkeypatch).context([desc], short) as ctx:
        ctx.set_state(0, fields, parts)
        st = _oracle_state(desc, fields, parts, arr)
        st.smooth_passes = smooth
        for nsteps in (1, 4):
            ctx.step(nsteps)
            oracle.step(st, nsteps)
            f, p, _ = ctx.get_state(0)
            _compare(desc, f, p, st, 1e-12, 1e-12 * max(shape), 1e-12)


@pytest.mark.parametrize("ndim,shape,bc", [(2, (33, 20, 1), 0), (3, (9, 11, 10), 1), (2, (1100, 900, 1), 0)])
def test_runs_of_one_context_with_and_without(monkeypatch, ndim, shape, bc):
    """The second run's planes are refused: the same states step alike in both, with energies,
    diagnostics, and momenta loaded in the presence of fields."""
    desc, fields, parts, _ = _case(ndim, shape, 0.05 if shape[0] > 1000 else 3, bc, 0, 410 + ndim)
    n = parts[0].shape[1]
    sort = 7 if shape[0] > 1000 else 0   # requests for the sort's scratch, which come last
    with _Allocator(monkeypatch).context([desc, desc], 1 + 2 * sort) as ctx:
        for r in range(2):
            ctx.set_state(r, fields, parts)
            ctx.load_maxwell_juttner(r, 0, n / np.prod(shape), 0.5, (0.1, 0.2, 0.0), seed=9)
        loaded = [ctx.get_state(r)[1][0] for r in range(2)]
        assert np.abs(loaded[0] - loaded[1]).max() <= 1e-14 * max(shape)
        ctx.step(5)
        (f0, p0, _), (f1, p1, _) = ctx.get_state(0), ctx.get_state(1)
        d0, d1 = ctx.diagnostics(0), ctx.diagnostics(1)
        h0, h1 = ctx.energy_history(0), ctx.energy_history(1)
    assert np.abs(f0 - f1).max() <= 1e-12 * np.abs(f0).max()
    for a, b in zip(p0, p1):
        d = np.abs(a - b)
        for x, L in zip(range(ndim), shape):
            d[x] = np.minimum(d[x], L - d[x])
        assert d.max() <= 1e-12 * max(shape)
    np.testing.assert_allclose(h0, h1, rtol=1e-11)
    np.testing.assert_allclose(d0["kinetic"], d1["kinetic"], rtol=1e-12)
    assert abs(d0["gauss_max"] - d1["gauss_max"]) <= 1e-12 * d0["rho_max"]


@pytest.mark.parametrize("ndim,small,large,sort", [(3, (64, 64, 64), (96, 96, 96), 6), (2, (400, 400, 1), (700, 700, 1), 0)])
def test_memory_per_cell_without(monkeypatch, ndim, small, large, sort):
    alloc, got = _Allocator(monkeypatch), []
    for shape in (small, large):   # (the larger grid's sort has requests of its own, after the planes')
        with alloc.context([pic.run_desc(ndim, *shape, 2.0, 8.0, 0.5, [(-1.0, 1.0, 100)])], 2 + (sort if shape == large else 0)):
            got.append(sum(alloc.sizes))
    staging = 8 * (np.prod(large) - np.prod(small))   # one plane, shared by all runs
    assert got[1] - got[0] - staging <= 120 * (np.prod(large) - np.prod(small))
