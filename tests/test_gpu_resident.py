"""The resident Leja kernel against one launch per term (EREM_TERM_LAG=1):
every cell takes the same operations in the same order, so the same schedules
and the same bits of T, at the edges of its blocks, vectors and tables."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu

# (dim, nx, ny, nz): one row, one cell, rows shorter than a vector, pitch
# remainders, one block, many blocks with a short last one, long rows, blocks
# in y and z, more than one vector per thread
SHAPES = [(2, 1, 1, 1), (2, 3, 7, 1), (2, 5, 1, 1), (2, 64, 64, 1), (2, 129, 305, 1), (2, 600, 470, 1),
          (2, 1023, 45, 1), (3, 4, 3, 2), (3, 33, 20, 9), (3, 16, 61, 50), (3, 70, 3, 41), (3, 50, 90, 40)]


def context(torch, monkeypatch, lag, dim, nx, ny, nz, prec, diag=False):
    monkeypatch.delenv("EREM_TERM_LAG", raising=False)
    if lag:
        monkeypatch.setenv("EREM_TERM_LAG", "1")
    n = nx * ny * nz
    rng = np.random.default_rng(nx + 1000 * ny + nz)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    one = np.ones(n)
    ramp = np.tile(1.0 - (np.arange(nx) + 0.5) / nx, ny * nz)
    # K of (y, z) only: the ramp is the pressure, the Leja copy has no
    # diagonal in FP32-bulk; a disturbed ramp keeps it
    lnk = np.repeat(rng.normal(0, 1, ny * nz), nx)
    if diag:
        ramp = ramp + 0.01 * rng.normal(0, 1, n)
    ctx = E.Context(dim, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision=prec)
    T = t(rng.uniform(20, 80, n))
    ctx.set_state(T, t(ramp), t(lnk), t(0.2 * one), t(one), 0.3 / max(nx, ny, nz))
    return ctx, T


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("diag", [False, True])
def test_resident_terms_have_the_bits_of_single_launches(monkeypatch, shape, prec, diag):
    torch = pytest.importorskip("torch")
    out = {}
    for lag in (0, 1):
        ctx, T = context(torch, monkeypatch, lag, *shape, prec, diag)
        dt = 0.3 / max(shape[1:])
        sch, runs = [], []
        for opts in (E.leja_opts(tol=1e-6), E.leja_opts(tol=1e-10), E.leja_opts(replay=[2, 1, 2])):
            try:  # some of the disturbed fluxes are too stiff for FP32: the same error then
                st = ctx.erem_step(T, dt, opts=opts)
            except E.EremError as e:
                assert e.status in (E.EREM_ENONFINITE, E.EREM_ENOTCONV)
                sch.append(e.status)
                continue
            sch.append(st.schedule)
            runs.append((st.launches, st.degree_total, st.err_est))
        out[lag] = (sch, T.cpu().numpy(), runs)
        ctx.close()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    for (l0, _, e0), (l1, m, e1) in zip(out[0][2], out[1][2]):
        assert l0 < l1 or m < 6          # the terms of a substep share a launch
        assert e0 == pytest.approx(e1, rel=1e-9)


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
def test_resident_terms_continue_over_several_launches(monkeypatch, prec):
    # a forced degree past the terms of one launch, and a free run past the
    # first table of divided differences
    torch = pytest.importorskip("torch")
    out = {}
    for lag in (0, 1):
        ctx, T = context(torch, monkeypatch, lag, 2, 70, 90, 1, prec)
        v = torch.linspace(-1.0, 1.0, 6300, dtype=torch.float64, device="cuda:0")
        r = []
        for opts in (E.leja_opts(replay=[1, 500]), E.leja_opts(tol=1e-7, m_max=400)):
            o = torch.zeros_like(v)
            try:  # q_m leaves the range of FP32 long before term 500: the same error then
                sch = ctx.phi1_apply(v, o, opts=opts).schedule
            except E.EremError as e:
                assert prec == "fp32_bulk" and e.status == E.EREM_ENONFINITE
                sch = e.status
            r.append((sch, o.cpu().numpy()))
        # steps of a halving length: from too stiff for 6 doublings (the same
        # error) through substeps to one substep, some past the first table
        degrees, T2 = [], T.clone()
        for k in range(12):
            try:
                sch = ctx.erem_step(T2, 0.35 * 0.5**k, opts=E.leja_opts(tol=1e-6, m_max=400)).schedule
                degrees += sch[1:]
            except E.EremError as e:
                assert e.status in (E.EREM_ENONFINITE, E.EREM_ENOTCONV)
                sch = e.status
            r.append((sch, T2.cpu().numpy()))
        assert prec == "fp32_bulk" or max(degrees) > 48
        # a window longer than the kernel's ring of estimates takes the launches
        st = ctx.erem_step(T2, 0.01, opts=E.leja_opts(avg_window=200))
        r.append((st.schedule, T2.cpu().numpy()))
        out[lag] = r
        ctx.close()
    for (s0, a0), (s1, a1) in zip(out[0], out[1]):
        assert s0 == s1 and np.array_equal(a0, a1)
