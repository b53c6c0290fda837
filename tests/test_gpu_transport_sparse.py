"""FP64 transport where the gas density is subnormal (37 scale heights up): 1/rho
overflows there, the Stokes number does not, and the particle must stay finite.

St is beyond 1e290, so the drift is 0 and what is left of r is the diffusion term
sqrt(2 D dt): r to 1e-12 as everywhere.  z settles to 1e-110 cm or less; its St carries
rho's subnormal rounding (2^-1075 over 1e-314: 3e-10), and z to 1e-2 allows for that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def test_subnormal_gas_densities():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()
    P = W.benchmark_disk()
    N = 256
    rng = np.random.default_rng(2)
    r = W.AU * rng.uniform(2.0, 50.0, N)
    z = rng.uniform(34.0, 37.45, N) * oracle.gas(P, r, np.zeros(N))["H"]
    rho = oracle.gas(P, r, z)["rho"]
    assert np.sum((rho > 1e-314) & (rho < 5e-309)) > 20 and np.sum(rho > 1e-270) > 20
    m, M, ids = np.full(N, 1e-11), np.full(N, 1e26), np.arange(N, dtype=np.uint32)
    s = oracle.DiskState(m, M, r, z, ids)
    oracle.transport(P, s, W.YR, seed=9, disk=0, step=0)
    ok = rho > 1e-314
    assert np.all(np.isfinite(s.r[ok]))
    d = mcd.Disk(P, (1, 1, N), seed=9, prec="fp64")
    mcd.mcd_set_particles(d.ctx, 0, m, M, r, z, ids)
    mcd.mcd_transport(d.ctx, W.YR)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    got = d.particles()
    d.close()
    assert np.all(np.abs(got["r"][ok] - s.r[ok]) <= 1e-12 * r[ok])
    assert np.all(np.abs(got["z"][ok] - s.z[ok]) <= 1e-2 * np.abs(s.z[ok]) + 1e-140)
