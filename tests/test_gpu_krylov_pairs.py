"""Bases of every remainder of the two-vectors-a-pass orthogonalisation against
the oracle's modified Gram-Schmidt, on forced substeps: 1e-11 or, if larger, 20
times the oracle's own response to a change of v by eps |J| |T|."""
import numpy as np
import pytest

import cases as C
import paper_1209_5553_gb300 as E
from oracle import krylov as K

pytestmark = pytest.mark.gpu

GRIDS = {"rect_37x23": lambda: C.heat2d_rect(37, 23), "box_9x7x5": lambda: C.random_case(3, 9, 7, 5, seed=3)}


@pytest.mark.parametrize("grid", list(GRIDS))
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 11, 32])
def test_bases_match_the_oracle(grid, m):
    torch = pytest.importorskip("torch")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    case = GRIDS[grid]()
    pb, g = case.problem(), case.grid
    J, v = pb.J(case.T0), pb.G(case.T0)
    yinf = float(np.max(np.abs(case.T0)))
    o = K.KrylovOptions(m=m, replay=[case.dt / 20, case.dt / 30, case.dt / 20])
    want = K.phi1_krylov(J, v, case.dt, yinf, o)
    rng = np.random.default_rng(m)
    scale = 2.0**-52 * (abs(J) @ np.abs(case.T0))
    resp = max(C.rel_l2(K.phi1_krylov(J, v + scale * rng.standard_normal(v.size), case.dt, yinf, o).value, want.value)
               for _ in range(3))
    with E.Context(g.dim, g.nx, g.ny, g.nz, physics=case.gpu_physics()) as ctx:
        ctx.set_state(t(case.T0), t(case.p), t(case.lnk), t(case.phi), t(case.lam), case.dt)
        out = t(np.zeros(case.n))
        st = ctx.phi1_apply_krylov(t(v), out, E.krylov_opts(m=m, replay=o.replay))
    assert st.dims[:3] == want.dims or list(st.dims[:3]) == list(want.dims)
    assert C.rel_l2(out.cpu().numpy(), want.value) < max(1e-11, 20 * resp)
