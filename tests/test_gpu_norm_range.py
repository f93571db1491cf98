"""||q_m||^2 beyond the range of FP32 in FP32-bulk: the Newton vectors of
converging interpolations pass 3.4e38 in their sum of squares where no cell's
square does, and every form of the terms has to go on there."""
import numpy as np
import pytest

import paper_1209_5553_gb300 as E

pytestmark = pytest.mark.gpu


def gauss(rng, ny, nx, sigma, ell):
    """Zero-mean Gaussian field of standard deviation sigma and correlation
    length ell on the unit square (periodic)."""
    f = np.fft.rfft2(rng.standard_normal((ny, nx)))
    k2 = (np.fft.rfftfreq(nx) * nx) ** 2 + ((np.fft.fftfreq(ny) * ny) ** 2)[:, None]
    x = np.fft.irfft2(f * np.exp(-((np.pi * ell) ** 2) * k2), s=(ny, nx))
    x -= x.mean()
    return (x * (sigma / x.std())).reshape(-1)


@pytest.mark.parametrize("cs", [0, 8])
def test_resident_members_keep_their_schedule(monkeypatch, cs):
    # strong permeability contrast: the norms of about one member in ten pass
    # 3.4e38 while the stopping test is still to be met, in one substep or in an
    # attempt that fails later.  k_ens_cluster sums in FP64.
    torch = pytest.importorskip("torch")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    sizes = [64, 75, 108, 141, 153, 164, 186, 197] * 6
    ph = E.Physics(100.0, 100.0, 1.0, 0.0, 80.0, 0)
    fields = []
    for e, n in enumerate(sizes):
        rng = np.random.default_rng(100 + e)
        lnk = t(gauss(rng, n, n, 1.5 + 0.2 * (e % 6), 0.1))
        x = (np.arange(n) + 0.5) / n
        p = t(np.tile(1.0 - x, n))
        with E.Context(2, n, n, physics=ph) as ctx:
            ctx.pressure_solve(lnk, None, p, tol=1e-12)
        T0 = 20.0 + 15.0 * np.repeat(x, n) + 3.0 * np.sin(6.28 * (rng.random() + np.tile(x, n)))
        fields.append((t(T0), p, lnk, t(np.full(n * n, 0.2)), t(np.full(n * n, 2.0))))
    out = {}
    for form in ("0", "1"):
        monkeypatch.setenv("EREM_ENS_RESIDENT", form)
        with E.Ensemble([(n, n, ph) for n in sizes], precision="fp32_bulk") as ens:
            for e, f in enumerate(fields):
                ens.set_member(e, *f, 0.05)
            ens.configure(E.leja_opts(tol=1e-6), cluster_ctas=cs)
            r = []
            for _ in range(2):   # the second run starts from the substeps of the first
                ens.run(2)
                for e, n in enumerate(sizes):
                    T = torch.empty(n * n, dtype=torch.float64, device="cuda:0")
                    ens.get_member(e, T)
                    st = ens.member_stats(e)
                    r.append((st.status, st.schedule, st.terms, st.attempts, T.cpu().numpy()))
            out[form] = r
    for a, b in zip(out["0"], out["1"]):
        assert a[:4] == b[:4]
        assert np.array_equal(a[4], b[4])
