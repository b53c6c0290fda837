"""The diagnostics' paths for large disks: moments in parts (above 16,384
particles; the part size grows with the number of bins) and the sigma map's
mass sum over many blocks, against the oracle.  Positions in zone order and
shuffled, particles on edges, repeated edges, removed particles, swarm masses
over twenty decades.  Both sides sum compensated: a few ulp of the largest
term, 1e-14, counts exactly, repeated calls the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
AU = W.AU


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("grid,nbins", [((16, 8, 128), 7), ((127, 1, 130), 1), ((127, 1, 130), 33), ((127, 1, 130), 227),
                                        ((61, 7, 157), 113), ((61, 7, 157), 1024)])
@pytest.mark.parametrize("shuffled", [0, 1])
def test_large_disk_diagnostics(grid, nbins, shuffled):
    N = grid[0] * grid[1] * grid[2]
    P = W.benchmark_disk()
    rng = np.random.default_rng(nbins)
    m, r, z = W.midrun_state(P, N, seed=nbins)
    M = 10.0 ** rng.uniform(10, 30, N)
    r[rng.random(N) < 0.03] = np.inf
    d = mcd.Disk(P, grid, seed=1, prec="mixed")
    mcd.mcd_set_particles(d.ctx, 0, m, M, r, z, np.arange(N, dtype=np.uint32))
    if not shuffled:
        mcd.mcd_regrid(d.ctx)
    x = d.particles()
    alive = np.sort(x["r"][np.isfinite(x["r"])])
    edges = np.sort(np.concatenate([np.geomspace(1.0, 90.0, nbins + 1 - (nbins + 1) // 3) * AU,
                                    rng.choice(alive, (nbins + 1) // 3)]))
    if nbins > 4:
        edges[3] = edges[2]
    got, want = d.moments(edges), oracle.moments(x["m"], x["M"], x["r"], edges)
    assert np.array_equal(got[:, 4], want[:, 4]) and want[:, 4].sum() > N // 2
    assert np.allclose(got, want, rtol=1e-14, atol=0.0)
    assert np.array_equal(d.moments(edges), got)
    me = np.geomspace(1e-11, 1e3, 40)
    smap, ref = d.sigma_map(edges, me), oracle.sigma_map(x["m"], x["M"], x["r"], edges, me)
    # each M is rounded to 2^-61 of the live mass: ten decades below the largest M stay exact to 1e-8 of themselves
    assert np.allclose(smap, ref, rtol=1e-12, atol=2.0**-60 * x["M"][np.isfinite(x["r"])].sum() * N)
    assert np.array_equal(d.sigma_map(edges, me), smap)
    d.close()
