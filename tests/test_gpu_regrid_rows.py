"""Whether a regrid's scatter CTAs add up their disk's groups of tiles themselves (two
launches per sort pass) or read them scanned (three): by the tiles times groups of all
disks together, so many mid-sized disks take the scan as one large disk does.  Ids,
columns and offsets equal the oracle's bit for bit on both sides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disks,launches", [(2, 12), (3, 16)])  # 625 tiles x 40 groups per disk; 65,536 rows
def test_rows_of_all_disks_decide(disks, launches):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()
    P, g = W.benchmark_disk(), (400, 16, 200)
    N = g[0] * g[1] * g[2]
    d = mcd.Disk([P] * disks, [g] * disks, seed=0, prec="mixed")
    rng = np.random.default_rng(1)
    cols = []
    for k in range(disks):
        m, r, z = W.midrun_state(P, N, seed=k)
        r[rng.random(N) < 0.01] = np.inf
        cols.append((m, np.full(N, 1e24), r, z, rng.permutation(N).astype(np.uint32)))
        mcd.mcd_set_particles(d.ctx, k, *cols[k])
    before = mcd.mcd_get_launch_count(d.ctx)
    mcd.mcd_regrid(d.ctx)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    assert mcd.mcd_get_launch_count(d.ctx) - before == launches
    for k in range(disks):
        s = oracle.DiskState(*cols[k])
        assert oracle.regrid(P, g[0], g[1], s)[0] == 0
        got = d.particles(k)
        assert np.array_equal(got["id"], s.id)
        for key in ("m", "M", "r", "z"):
            assert np.array_equal(got[key].view(np.uint64), getattr(s, key).view(np.uint64)), key
    d.close()
