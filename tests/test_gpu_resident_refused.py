"""A device that cannot run all CTAs of the resident Leja kernel at once (fewer
SMs than it reports, as in a partitioned context) refuses the launch: the step
then takes one launch per term.  Planning for more SMs than there are
(EREM_RES_SMS) has the driver refuse it in the same way."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E
from test_gpu_tape_limits import Problem, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
def test_refused_launch_falls_back_to_single_terms(monkeypatch, prec):
    torch = pytest.importorskip("torch")
    if torch.cuda.get_device_properties(0).multi_processor_count >= 160:
        pytest.skip("runs 160 CTAs at once")
    nx, ny = 256, 160   # one row to a CTA, 160 of them
    n = nx * ny
    rng = np.random.default_rng(9)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    x = np.tile((np.arange(nx) + 0.5) / nx, ny)
    fields = (t(1.0 - x), t(np.repeat(rng.normal(0, 1, ny), nx)), t(np.full(n, 0.2)), t(np.ones(n)))
    T0 = t(rng.uniform(20, 80, n))
    out = {}
    for name, value in (("EREM_RES_SMS", None), ("EREM_RES_SMS", "160"), ("EREM_TERM_LAG", "1")):
        monkeypatch.delenv("EREM_RES_SMS", raising=False)
        if value:
            monkeypatch.setenv(name, value)
        with E.Context(2, nx, ny, physics=E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0), precision=prec) as ctx:
            ctx.set_state(T0, *fields, 0.002)
            T = T0.clone()
            st = [ctx.erem_step(T, 0.002) for _ in range(3)]
            out[name, value] = ([s.schedule for s in st], [s.launches for s in st], T.cpu().numpy())
    res, refused, single = out.values()
    assert refused[0] == single[0] == res[0]
    assert np.array_equal(refused[2], single[2]) and np.array_equal(res[2], single[2])
    assert refused[1][1:] == single[1][1:] and res[1][1] < single[1][1]


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
def test_refused_launch_of_a_taped_step(monkeypatch, prec):
    torch = pytest.importorskip("torch")
    if torch.cuda.get_device_properties(0).multi_processor_count >= 160:
        pytest.skip("runs 160 CTAs at once")

    class Rows(Problem):
        nx, ny, n = 142, 160, 142 * 160   # fp32_bulk: one row to a CTA (36 vectors)

    pr = Rows(torch, prec)
    pr.qbytes = 144 * pr.ny * (4 if prec == "fp32_bulk" else 8)
    dt = 0.002
    ref = pr.run(dt)
    monkeypatch.setenv("EREM_RES_SMS", "160")
    same(pr.run(dt, 400), ref)
    same(pr.run(dt), ref)
    sch = ref[0]
    same(pr.run(dt, sum(sch[1:]) + 2 * len(sch), replay=sch), ref)
