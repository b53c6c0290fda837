"""Transport over the gas slopes and both settling forms, against the oracle.

FP64 forms slopes that are multiples of one half up to 4 by products and all others by
pow; the displacements hold to 1e-12 (1e-5 in the mixed path) of the step and the
diffusion length, as for the benchmark disk's slopes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
AU, YR = W.AU, W.YR
TOL = {"fp64": 1e-12, "mixed": 1e-5}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("p,q", [(0.0, 0.0), (1.5, 0.5), (1.5, 3.0 / 7.0), (0.9, 0.43), (4.0, 1.0), (0.75, 4.0), (4.5, 0.5),
                                 (-0.5, 0.25)])
def test_transport_slopes(prec, form, p, q):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()
    P = W.benchmark_disk(p=p, q=q, settle_form=form)
    N = 8 * 4 * 60
    rng = np.random.default_rng(4)
    r = rng.uniform(1.2 * P["r_in"], 0.95 * P["r_out"], N)
    z = rng.normal(0, 1, N) * oracle.gas(P, r, np.zeros(N))["H"]
    m, M, ids = W.random_masses(N, seed=5, lo=1e-12, hi=1e4), np.full(N, 3e26), rng.permutation(N).astype(np.uint32)
    d = mcd.Disk(P, (8, 4, 60), seed=9, prec=prec)
    mcd.mcd_set_particles(d.ctx, 0, m, M, r, z, ids)
    mcd.mcd_transport(d.ctx, YR)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    got = d.particles()
    d.close()
    s = oracle.DiskState(m, M, r, z, ids)
    oracle.transport(P, s, YR, seed=9, disk=0, step=0)
    keep = np.isfinite(s.r)
    assert np.array_equal(keep, np.isfinite(got["r"])) and keep.sum() > N // 2
    sig = np.sqrt(2 * oracle.gas(P, r[keep], z[keep])["D"] * YR)
    for k, x0 in (("r", r), ("z", z)):
        x, o, x0 = got[k][keep], getattr(s, k)[keep], x0[keep]
        assert np.all(np.abs(x - o) <= TOL[prec] * (np.abs(o - x0) + sig) + 1e-15 * np.abs(x0)), k
