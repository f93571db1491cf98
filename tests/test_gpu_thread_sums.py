"""The range of ||q_m||^2 in FP32-bulk: the forms of the Leja terms that give a
thread many cells (a block that stays on the chip, a march through the planes)
accept at least what the launches term by term accept."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


# a block of four vectors per thread; a march of pairs, with and without the
# diagonal
@pytest.mark.parametrize("shape, diag", [((2, 1024, 1024, 1), False), ((2, 1024, 1024, 1), True),
                                         ((3, 96, 128, 128), False), ((3, 96, 128, 128), True)])
def test_a_threads_sum_keeps_the_range_of_its_squares(monkeypatch, shape, diag):
    torch = pytest.importorskip("torch")
    dim, nx, ny, nz = shape
    n = nx * ny * nz
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    # a problem that is linear in T (no inflow temperature), T alternating in y and
    # z and uniform in x: the cells' squares are alike, and a scale of T carries a
    # thread's sum of them past FP32 before any of them
    sign = (-1.0) ** (np.arange(nz)[:, None, None] + np.arange(ny)[None, :, None])
    T0 = t((20.0 + 60.0 * sign * np.ones((1, 1, nx))).reshape(-1))
    ramp = np.tile(1.0 - (np.arange(nx) + 0.5) / nx, ny * nz)
    if diag:   # a disturbed ramp keeps the diagonal of the Leja copy
        ramp = ramp + 1e-6 * np.random.default_rng(3).normal(0, 1, n)
    one = np.ones(n)
    dt = 0.3 / max(shape[1:])
    step = {}
    for lag in (0, 1):
        monkeypatch.delenv("EREM_TERM_LAG", raising=False)
        if lag:
            monkeypatch.setenv("EREM_TERM_LAG", "1")
        ctx = E.Context(dim, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 0.0, 0), precision="fp32_bulk")
        ctx.set_state(T0, t(ramp), t(0.0 * one), t(0.2 * one), t(one), dt)

        def run(scale, ctx=ctx):
            T = scale * T0
            try:
                return ctx.erem_step(T, dt).schedule, T
            except E.EremError as e:
                assert e.status in (E.EREM_ENONFINITE, E.EREM_ENOTCONV)
                return None, T

        step[lag] = run
    substeps = lambda r: r[0][0] if r[0] else 1000
    least = substeps(step[1](2.0**20))
    assert least < 1000
    # the first power of two at which the launches need more substeps
    edge = next(k for k in range(24, 80) if substeps(step[1](2.0**k)) > least)
    for j in range(-16, 17):
        a, b = step[1](2.0 ** (edge + j / 8)), step[0](2.0 ** (edge + j / 8))
        assert substeps(b) <= substeps(a), (edge, j)
        if a[0] and a[0] == b[0]:
            assert torch.equal(a[1], b[1]), (edge, j)
