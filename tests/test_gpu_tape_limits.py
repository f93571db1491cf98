"""Taped steps at the limits of their arena: whatever of an interpolation fits,
T and the gradient have the bits of an untaped step."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


class Problem:
    """70 x 90 (all terms of a substep in one launch), layers along x and a
    step that takes one substep of more than 48 terms (the first table)."""

    nx, ny = 70, 90
    n = nx * ny
    m_max = 150

    def __init__(self, torch, prec):
        self.torch, self.prec = torch, prec
        self.qbytes = 72 * self.ny * (4 if prec == "fp32_bulk" else 8)   # rows of 72 cells
        rng = np.random.default_rng(7)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
        x = (np.arange(self.nx) + 0.5) / self.nx
        depth = (np.arange(self.ny) + 0.5) / self.ny
        self.T0 = t((20.0 + 15.0 * depth[:, None] + 3.0 * np.sin(6.28 * x)[None, :]).reshape(-1))
        self.fields = (t(np.tile(1.0 - x, self.ny)), t(np.repeat(rng.normal(0, 1, self.ny), self.nx)),
                       t(np.full(self.n, 0.2)), t(np.full(self.n, 1.0)))
        self.lam = t(rng.normal(0, 1, self.n))

    def context(self, dt):
        ctx = E.Context(2, self.nx, self.ny, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision=self.prec)
        ctx.set_state(self.T0, *self.fields, dt)
        return ctx

    def run(self, dt, vectors=None, **opts):
        """(schedule, T, lambda after the adjoint of the step); vectors: the
        arena's room in Newton vectors, None without a tape."""
        with self.context(dt) as ctx:
            if vectors is not None:
                ctx.adjoint_tape(int(vectors * self.qbytes), True)
            T = self.T0.clone()
            sch = ctx.erem_step(T, dt, opts=E.leja_opts(**opts)).schedule
            lam = self.lam.clone()
            ctx.adjoint_begin()
            ctx.adjoint_step(self.T0, lam, sch)
            return sch, T.cpu().numpy(), lam.cpu().numpy()

    def long_step(self):
        """A step length whose first attempt needs between 52 and 140 terms."""
        for k in range(24):
            dt = 0.2 * 0.75**k
            try:
                sch = self.run(dt, tol=1e-6)[0]
            except E.EremError:
                continue
            if len(sch) == 2 and 52 <= sch[1] <= 140:
                return dt
        raise AssertionError("no step of one long substep")


def same(a, b):
    assert a[0] == b[0]
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
def test_a_step_that_outgrows_its_tape(monkeypatch, prec):
    # the arena holds the terms of the first table (49 vectors, 51 with the
    # two that complete P) but not always those of the full one (151, 153)
    torch = pytest.importorskip("torch")
    pr = Problem(torch, prec)
    monkeypatch.delenv("EREM_TERM_LAG", raising=False)
    dt = pr.long_step()
    ref = pr.run(dt, tol=1e-6)
    for vectors in (48, 49, 50, 51, 60, 100, 150, 151, 152, 153, 154, 400):
        same(pr.run(dt, vectors, tol=1e-6), ref)
    monkeypatch.setenv("EREM_TERM_LAG", "1")   # one launch per term
    same(pr.run(dt, tol=1e-6), ref)
    same(pr.run(dt, 60, tol=1e-6), ref)


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
def test_full_tape_of_one_long_step(prec):
    # MisfitModel(tape="full") reserves 64 vectors for each step and one more
    torch = pytest.importorskip("torch")
    from paper_1209_5553_gb300.autograd import MisfitModel, misfit

    pr = Problem(torch, prec)
    dt = pr.long_step()
    obs = torch.arange(0, pr.n, 97, device="cuda:0")
    data = torch.full((len(obs),), 30.0, dtype=torch.float64, device="cuda:0")
    out = {}
    for tape in (False, "full"):
        m = MisfitModel(2, pr.nx, pr.ny, 1, E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), pr.fields[2], pr.fields[3], dt,
                        1, obs, data, precision=prec, tape=tape)
        lnk = pr.fields[1].clone().requires_grad_(True)
        T0 = pr.T0.clone().requires_grad_(True)
        L = misfit(lnk, T0, m)
        g = torch.autograd.grad(L, [lnk, T0])
        out[tape] = (m.schedules, float(L.detach()), g[0].cpu().numpy(), g[1].cpu().numpy())
        m.close()
    a, b = out[False], out["full"]
    assert a[0] == b[0] and a[0][0][1] > 48
    assert a[1] == b[1]
    assert np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("degree", [237, 238, 239, 240, 241, 479, 480])
def test_forced_degrees_at_the_end_of_a_launch(degree):
    # a launch takes 240 terms; the arena holds the q_0 .. q_degree of this
    # step and nothing more (FP32's range ends before such degrees)
    torch = pytest.importorskip("torch")
    pr = Problem(torch, "fp64")
    dt = pr.long_step()
    same(pr.run(dt, degree + 1, replay=[1, degree]), pr.run(dt, replay=[1, degree]))
