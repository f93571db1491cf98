"""Waits inside the Leja kernels that run out: the step fails with its own
status, the state and the device stay usable.  EREM_WAIT_POLLS=0 gives up every
wait at once (the messages and copies waited for still arrive)."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


# terms on the chip, one and several vectors per thread; pairs of terms on grids
# whose blocks march through few and many planes
@pytest.mark.parametrize("shape, prec", [((2, 64, 64, 1), "fp64"), ((2, 700, 600, 1), "fp32_bulk"),
                                         ((3, 40, 40, 40), "fp64"), ((3, 96, 128, 128), "fp32_bulk"),
                                         ((3, 128, 130, 100), "fp32_bulk")], ids=str)
def test_a_wait_that_runs_out_is_an_error(monkeypatch, shape, prec):
    torch = pytest.importorskip("torch")
    dim, nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(5)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    x = np.tile((np.arange(nx) + 0.5) / nx, ny * nz)
    fields = (t(1.0 - x), t(np.repeat(rng.normal(0, 1, ny * nz), nx)), t(np.full(n, 0.2)), t(np.ones(n)))
    T0 = t(rng.uniform(20, 80, n))
    dt = 0.3 / max(shape[1:])

    def step(polls):
        monkeypatch.delenv("EREM_WAIT_POLLS", raising=False)
        if polls is not None:
            monkeypatch.setenv("EREM_WAIT_POLLS", str(polls))
        with E.Context(dim, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision=prec) as ctx:
            ctx.set_state(T0, *fields, dt)
            T, err = T0.clone(), []
            for _ in range(2):
                try:
                    ctx.erem_step(T, dt)
                except E.EremError as e:
                    err.append(e.status)
            torch.cuda.synchronize()
            return T, err

    ref, none = step(None)
    assert not none
    T, err = step(0)
    assert err == [E.EREM_ETIMEOUT] * 2 and torch.equal(T, T0)
    again, none = step(None)
    assert not none and torch.equal(again, ref)


@pytest.mark.parametrize("shape, prec", [((2, 64, 64, 1), "fp64"), ((3, 96, 128, 128), "fp32_bulk")], ids=str)
def test_the_message_names_no_other_kernel(monkeypatch, shape, prec):
    torch = pytest.importorskip("torch")
    dim, nx, ny, nz = shape
    n = nx * ny * nz
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    x = np.tile((np.arange(nx) + 0.5) / nx, ny * nz)
    monkeypatch.setenv("EREM_WAIT_POLLS", "0")
    with E.Context(dim, nx, ny, nz, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision=prec) as ctx:
        T = t(20.0 + 15.0 * x)
        ctx.set_state(T, t(1.0 - x), t(np.zeros(n)), t(np.full(n, 0.2)), t(np.ones(n)), 0.002)
        with pytest.raises(E.EremError, match="wait") as err:
            ctx.erem_step(T, 0.002)
    assert "resident" not in str(err.value)
