"""Host time of an ensemble run: the split of the members into launches is made
once and kept while their passes per step stay about the same."""
import time

import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


def test_planned_runs_cost_the_host_no_more_than_fixed_ones():
    # 600 members, one step a run: played through anew, the candidates' queues take
    # several times as long as all the other host work of a run (which the run on
    # clusters of a given size has too)
    torch = pytest.importorskip("torch")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    ph = E.Physics(50.0, 40.0, 1.0, 0.0, 80.0, 0)
    sizes = [8 + e % 9 for e in range(600)]
    host = {}
    with E.Ensemble([(n, n, ph) for n in sizes], precision="fp32_bulk") as ens:
        rng = np.random.default_rng(1)
        for e, n in enumerate(sizes):
            x = np.tile((np.arange(n) + 0.5) / n, n)
            ens.set_member(e, t(20.0 + 15.0 * x), t(1.0 - x), t(np.repeat(rng.normal(0, 1, n), n)),
                           t(np.full(n * n, 0.2)), t(np.ones(n * n)), 0.005)
        for cs in (8, 0):
            ens.configure(E.leja_opts(tol=1e-6), cluster_ctas=cs)
            for _ in range(4):
                ens.run(1)
            times = []
            for _ in range(15):
                t0 = time.perf_counter()
                st = ens.run(1)
                times.append(time.perf_counter() - t0 - 1e-3 * st.t_ms)
            host[cs] = sorted(times)[len(times) // 2]
    assert host[0] < 1.5 * host[8] + 1e-4, host
