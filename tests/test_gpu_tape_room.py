"""The arena a taped step needs: the Newton vectors of its table (q_0 .. q_M),
the same for the resident form of the terms, which runs two terms past it."""
import numpy as np
import pytest

from test_gpu_tape_limits import Problem

pytestmark = pytest.mark.gpu


def gradient(pr, dt, vectors):
    """d/d ln K of lam . T after one step taped into an arena of so many Newton
    vectors.  The adjoint is handed a state other than the step's: a taped step's
    Newton vectors are still those of T0, recomputed ones are not."""
    torch = pr.torch
    with pr.context(dt) as ctx:
        if vectors:
            ctx.adjoint_tape(vectors * pr.qbytes, True)
        T = pr.T0.clone()
        sch = ctx.erem_step(T, dt).schedule
        lam = pr.lam.clone()
        ctx.adjoint_begin()
        ctx.adjoint_step(pr.T0 * 1.5 + torch.sin(pr.T0), lam, sch)
        g = torch.zeros_like(lam)
        ctx.adjoint_lnk(pr.fields[1], g)
        return sch, g.cpu().numpy()


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
@pytest.mark.parametrize("length", ["short", "long"])
def test_arena_of_one_table_tapes_the_step(prec, length):
    torch = pytest.importorskip("torch")
    pr = Problem(torch, prec)
    dt = pr.long_step()
    if length == "short":
        while pr.run(dt)[0][1] > 44:
            dt *= 0.7
    need = 49 if length == "short" else pr.m_max + 1   # the first table, or the full one
    sch, taped = gradient(pr, dt, 400)
    assert len(sch) == 2 and (sch[1] <= 48) == (length == "short")
    assert not np.array_equal(taped, gradient(pr, dt, 0)[1])
    assert np.array_equal(taped, gradient(pr, dt, need)[1])
