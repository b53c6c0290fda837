"""Which path the moments take: parts of consecutive slots (two launches) where a
part holds few bins, one CTA per bin (one launch) for small disks and for many
bins, on both sides of each line, against the oracle.  Both sum compensated: a few
ulp of the largest term, 1e-14; counts exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,nbins,launches", [
    ((16, 8, 128), 1, 1), ((127, 1, 130), 1, 2),           # 16,384 particles, and more
    ((127, 1, 130), 10, 2), ((127, 1, 130), 11, 1),        # 1,536 particles per bin
    ((64, 8, 136), 45, 2), ((64, 8, 136), 46, 1), ((64, 8, 136), 1024, 1),
    ((57, 16, 256), 113, 2),                               # parts of 1,024
    ((57, 16, 256), 114, 2), ((57, 16, 256), 115, 1)])     # larger parts: 2,048 particles per bin
def test_moments_path_by_particles_per_bin(grid, nbins, launches):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()
    N = grid[0] * grid[1] * grid[2]
    P = W.benchmark_disk()
    m, r, z = W.midrun_state(P, N, seed=nbins)
    M = 10.0 ** np.random.default_rng(nbins).uniform(20, 26, N)
    d = mcd.Disk(P, grid, seed=1, prec="mixed")
    mcd.mcd_set_particles(d.ctx, 0, m, M, r, z, np.arange(N, dtype=np.uint32))
    edges = np.geomspace(1.0, 100.0, nbins + 1) * W.AU
    for ordered in (0, 1):
        if ordered:
            mcd.mcd_regrid(d.ctx)
        x = d.particles()
        before = mcd.mcd_get_launch_count(d.ctx)
        got = d.moments(edges)
        assert mcd.mcd_get_launch_count(d.ctx) - before == launches
        want = oracle.moments(x["m"], x["M"], x["r"], edges)
        assert np.array_equal(got[:, 4], want[:, 4])
        assert np.allclose(got, want, rtol=1e-14, atol=0.0)
    d.close()
