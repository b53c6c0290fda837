"""FP64 transport's vertical step over the whole range of k dt, against the oracle.

z0 exp(-k dt) has to keep its relative accuracy however much of z0 is left.  With
alpha = 1e-60 diffusion adds 1e-30 of a scale height; where that is what is left, it
holds to 1e-13.  exp amplifies the roundings of its argument by k dt: St passes some
fifteen operations on either side, one of them a slope of up to 4, so k dt holds to
1e-14 with a margin of two, and z to 1e-14 (1 + k dt).  Slopes that are multiples of
one half (products) and others (pow), and both settling forms, take the same step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
AU, YR = W.AU, W.YR


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()


def _step(P, m, r, z, dt):
    N = m.size
    d = mcd.Disk(P, (1, N // 64, 64), seed=9, prec="fp64")
    ids = np.arange(N, dtype=np.uint32)
    mcd.mcd_set_particles(d.ctx, 0, m, np.full(N, 3e26), r, z, ids)
    mcd.mcd_transport(d.ctx, dt)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    got = d.particles()
    d.close()
    s = oracle.DiskState(m, np.full(N, 3e26), r, z, ids)
    oracle.transport(P, s, dt, seed=9, disk=0, step=0)
    return got, s


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("p,q", [(1.0, 0.5), (1.5, 3.0 / 7.0), (0.0, 0.0), (4.0, 4.0), (0.9, 0.5), (-0.5, 0.43)])
def test_settled_height_keeps_its_digits(p, q, form):
    P = W.benchmark_disk(p=p, q=q, settle_form=form, alpha=1e-60, tr_flags=W.TR_VERTICAL)
    rng = np.random.default_rng(4)
    N = 64 * 64
    r = AU * np.exp(rng.uniform(0.0, np.log(30.0), N))
    z = rng.choice([-1.0, 1.0], N) * rng.uniform(0.1, 1.0, N) * oracle.gas(P, r, np.zeros(N))["H"]
    # masses of a Stokes number that gives k dt = x, from the Epstein law
    x = np.exp(rng.uniform(np.log(1e-6), np.log(100.0), N))
    x[:6] = [0.5 * (1 - 1e-9), 0.5 * (1 + 1e-9), 5.0, 10.0, 20.0, 40.0]
    g = oracle.gas(P, r, z)
    dt = 20.0 * YR * (30.0 if form else 1.0)
    St = np.minimum(x / (g["Omega"] * dt), 1e3)
    a = St * g["rho"] * g["vth"] / (P["rho_s"] * g["Omega"])
    m = 4.0 / 3.0 * np.pi * P["rho_s"] * a**3
    got, s = _step(P, m, r, z, dt)
    St = np.array([oracle.particle(P, r[k], z[k], m[k:k + 1])[1][0] for k in range(N)])
    x = g["Omega"] * (St / (1 + St) if form else St) * dt
    assert x.min() < 1e-5 and x.max() > 50.0
    assert np.all(np.abs(got["z"] - s.z) <= 1e-14 * (1 + x) * np.abs(s.z) + 1e-13 * np.abs(s.z - z * np.exp(-x)))
    assert np.array_equal(got["r"], r)
