"""The small multigrid levels in one launch against a launch per operation
(EREM_MG_SMALL=0): the same operations in the same order, so the same
iterations and the same bits, at the edges of the coarsening."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu

# (dim, nx, ny, nz): one coarse level, rows and columns, odd sizes, the largest
# small level, levels above it, prime sizes
SHAPES = [(2, 7, 5, 1), (2, 300, 1, 1), (2, 1, 257, 1), (2, 64, 64, 1), (2, 129, 127, 1), (2, 301, 203, 1),
          (3, 9, 1, 40), (3, 17, 33, 5), (3, 32, 32, 32), (3, 61, 37, 43)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_small_levels_have_the_bits_of_launches(monkeypatch, shape):
    torch = pytest.importorskip("torch")
    dim, nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(n)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    lnk, one = t(rng.normal(0, 1.5, n)), t(np.ones(n))
    T0 = rng.uniform(20, 80, n)
    out = {}
    for v in ("1", "0"):
        monkeypatch.setenv("EREM_MG_SMALL", v)
        r = []
        with E.Context(dim, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0)) as ctx:
            ctx.set_pressure_precond(0)
            for nu in (3, 1, 2, 5):
                ctx.set_pressure_multigrid(nu, 1.8)
                p = t(np.zeros(n))
                st = ctx.pressure_solve(lnk, None, p, tol=1e-10, maxit=2000)
                r += [st.lin_iters, p.cpu().numpy()]
            T = t(T0)
            st = ctx.rosm_step(T, 0.02, E.EREM_ROS2, p, lnk, 0.2 * one, one, lin_tol=1e-10, maxit=2000)
            r += [st.lin_iters, T.cpu().numpy()]
        out[v] = r
    for a, b in zip(out["1"], out["0"]):
        assert np.array_equal(a, b)
