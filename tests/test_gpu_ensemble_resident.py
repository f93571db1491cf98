"""The resident ensemble kernel against the one that works from L2
(EREM_ENS_RESIDENT=0): the same operations per cell in the same order, so the
same schedules and the same bits, at the edges of bands, vectors and clusters
and for runs split over several launches."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu

# fewer rows than CTAs, one row, rows shorter than a vector, pitch remainders, a
# short last band, sizes of every class (the last fits on no cluster)
SIZES = [(5, 9), (33, 1), (3, 40), (64, 64), (65, 67), (130, 97), (201, 190), (300, 310), (410, 400)]


def run(torch, prec, cs, diag):
    rng = np.random.default_rng(3)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    ph = E.Physics(100.0, 80.0, 1.0, 0.0, 80.0, 0)
    with E.Ensemble([(nx, ny, ph) for nx, ny in SIZES], precision=prec) as ens:
        for e, (nx, ny) in enumerate(SIZES):
            n = nx * ny
            ramp = np.tile(1.0 - (np.arange(nx) + 0.5) / nx, ny)
            if diag:   # not divergence-free: the Leja copy keeps its diagonal
                ramp = ramp + 1e-5 * rng.normal(0, 1, n)
            lnk = np.repeat(rng.normal(0, 0.3, ny), nx)
            ens.set_member(e, t(rng.uniform(20, 80, n)), t(ramp), t(lnk), t(np.full(n, 0.2)), t(np.full(n, 2.0)),
                           4.0 / max(nx, ny) ** 2 if diag else 2.0 / max(nx, ny, 8))
        ens.configure(E.leja_opts(tol=1e-6), cluster_ctas=cs)
        ens.run(2)
        ens.run(1)
        out = []
        for e, (nx, ny) in enumerate(SIZES):
            T = torch.empty(nx * ny, dtype=torch.float64, device="cuda:0")
            ens.get_member(e, T)
            st = ens.member_stats(e)
            out.append((st.status, st.steps_done, st.schedule, st.terms, st.passes, T.cpu().numpy()))
        return out


@pytest.mark.parametrize("prec", ["fp64", "fp32_bulk"])
@pytest.mark.parametrize("cs", [0, 2, 16])
@pytest.mark.parametrize("diag", [False, True])
def test_resident_members_have_the_bits_of_the_l2_kernel(monkeypatch, prec, cs, diag):
    torch = pytest.importorskip("torch")
    monkeypatch.setenv("EREM_ENS_RESIDENT", "0")
    ref = run(torch, prec, cs, diag)
    monkeypatch.setenv("EREM_ENS_RESIDENT", "1")
    got = run(torch, prec, cs, diag)
    for a, b in zip(got, ref):
        assert a[:5] == b[:5]
        assert np.array_equal(a[5], b[5])
