"""Two Leja terms per pass (EREM_TERM_PAIR=1) against one launch per term
(EREM_TERM_LAG=0): every cell takes the same operations in the same order, so
the same schedules and the same bits of T, at the edges of its blocks."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu

# (nx, ny, nz): one plane, two planes, one row, one cell, pitch remainders, rows that
# end inside a tile of 128 cells, blocks with short last rows and planes, wide
# rows (few to a block), many rows to a block
SHAPES = [(8, 9, 1), (7, 5, 2), (33, 1, 9), (1, 1, 3), (20, 31, 17), (100, 37, 29), (128, 40, 33), (130, 64, 21),
          (256, 30, 40), (381, 23, 18), (12, 300, 25), (60, 80, 150)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("diag", [False, True])
def test_pairs_have_the_bits_of_single_terms(monkeypatch, shape, diag):
    torch = pytest.importorskip("torch")
    nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(nx + 1000 * ny + nz)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    one = np.ones(n)
    ramp = np.tile(1.0 - (np.arange(nx) + 0.5) / nx, ny * nz)
    lnk = np.repeat(rng.normal(0, 1, ny * nz), nx)   # K of (y, z): the ramp is the pressure
    T0 = rng.uniform(20, 80, n)
    T0[: n // 3] = 20.0                              # zeros and subnormals in q_m
    out = {}
    for form in ("EREM_TERM_PAIR", "EREM_TERM_LAG"):
        for v in ("EREM_TERM_PAIR", "EREM_TERM_LAG"):
            monkeypatch.delenv(v, raising=False)
        monkeypatch.setenv(form, "1" if form == "EREM_TERM_PAIR" else "0")
        monkeypatch.setenv("EREM_LEJA_DIAG", "1" if diag else "0")
        ctx = E.Context(3, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision="fp32_bulk")
        T, dt = t(T0), 0.3 / max(shape)
        ctx.set_state(T, t(ramp), t(lnk), t(0.2 * one), t(one), dt)
        r = []
        # odd and even degrees, a forced odd degree, one and two terms
        for o in (dict(tol=1e-6), dict(tol=1e-5), dict(tol=1e-4), dict(replay=[2, 7, 1]), dict(replay=[1, 2]),
                  dict(tol=1e-6, m_max=5, max_doublings=6)):
            try:
                st = ctx.erem_step(T, dt, opts=E.leja_opts(**o))
            except E.EremError as e:     # the same error on both sides
                r.append((e.status, T.cpu().numpy()))
                continue
            r.append((st.schedule, T.cpu().numpy()))
            last = st
        out[form] = (r, last.err_est)
        ctx.close()
    (a, ea), (b, eb) = out["EREM_TERM_PAIR"], out["EREM_TERM_LAG"]
    for (s0, x0), (s1, x1) in zip(a, b):
        assert s0 == s1
        assert np.array_equal(x0, x1)
    assert ea == pytest.approx(eb, rel=1e-9)
