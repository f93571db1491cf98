"""A stage solve after the pressure preconditioner has changed: the pressure and
stage iteration graphs are kept apart, each for its own key."""
import numpy as np
import pytest

import cases as C
import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [1, 2, 4])
def test_stage_graph_outlives_a_new_pressure_graph(nu):
    torch = pytest.importorskip("torch")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    case = C.random_case(2, 41, 33, seed=nu, fluid_model=0)
    fields = [t(a) for a in (case.p, case.lnk, case.phi, case.lam)]
    g = case.grid
    with E.Context(2, g.nx, g.ny, physics=case.gpu_physics()) as ctx:
        ctx.set_pressure_precond(0)
        out = []
        for mg_nu in (3, nu):
            ctx.set_pressure_multigrid(mg_nu, 1.8)
            p = t(np.zeros(g.n))
            ctx.pressure_solve(fields[1], None, p, tol=1e-10, maxit=500)
            T = t(case.T0)
            ctx.rosm_step(T, 0.05, E.EREM_ROS2, *fields, lin_tol=1e-10, maxit=500)
            out.append(T.cpu().numpy())
    assert np.array_equal(out[0], out[1])
