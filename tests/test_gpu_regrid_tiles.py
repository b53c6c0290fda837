"""The radial sort's tiles and groups of tiles against the oracle's regrid.

A sort pass counts digits per tile (2,048 particles) and per group of 16 tiles;
tiles and groups belong to one disk.  Sizes at the edges of both, one disk
beyond 64 groups (2,097,152 particles), where the groups' counts are scanned
by a launch of their own, and several disks of unequal size in one context,
below and beyond that.  Radii over the disk and, as the worst case for the
digit counts, all in a few runs of equal upper words.  Ids, columns, offsets,
bounds and volumes must equal the oracle's bit for bit, twice in a row."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()


def _state(P, N, seed, narrow):
    rng = np.random.default_rng(seed)
    m, r, z = W.midrun_state(P, N, seed=seed)
    if narrow:
        r = P["r_in"] * (1.0 + 1e-7 * rng.integers(1, 40, N)) * 2.0
        z = rng.normal(0, 0.03, N) * r
    r[rng.random(N) < 0.01] = np.inf
    return m, 10.0 ** rng.uniform(20, 26, N), r, z, rng.permutation(N).astype(np.uint32)


@pytest.mark.parametrize("grids", [
    [(1, 1, 1)], [(23, 1, 89)], [(16, 4, 32)], [(683, 1, 3)],       # 1; 2,047; one tile; one more
    [(31, 7, 151)], [(64, 8, 64)], [(11, 9, 331)],                  # 32,767; one group; one more
    [(512, 16, 256)], [(1025, 16, 128)],                            # 64 groups; a 65th
    [(16, 4, 32), (11, 9, 331), (683, 1, 3), (64, 8, 64)],
    [(683, 1, 3), (1025, 16, 128), (11, 9, 331)]], ids=str)
@pytest.mark.parametrize("narrow", [0, 1])
def test_tiles_and_groups_match_the_oracle(grids, narrow):
    P = W.benchmark_disk()
    d = mcd.Disk([P] * len(grids), grids, seed=0, prec="mixed")
    want = []
    for k, g in enumerate(grids):
        cols = _state(P, g[0] * g[1] * g[2], 10 + k, narrow and g[0] * g[1] * g[2] < 40000)
        mcd.mcd_set_particles(d.ctx, k, *cols)
        s = oracle.DiskState(*cols)
        st, _, off, cb, cv, na = oracle.regrid(P, g[0], g[1], s)
        assert st == 0
        want.append((s, off, cb, cv))
    for _ in range(2):
        mcd.mcd_regrid(d.ctx)
        assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
        for k, (g, (s, off, cb, cv)) in enumerate(zip(grids, want)):
            got = d.particles(k)
            assert np.array_equal(got["id"], s.id)
            for key in ("m", "M", "r", "z"):
                assert np.array_equal(got[key].view(np.uint64), getattr(s, key).view(np.uint64)), key
            C = g[0] * g[1]
            goff, gb, gv = np.zeros(C + 1, np.int64), np.zeros((C, 6)), np.zeros(C)
            mcd.mcd_get_cells(d.ctx, k, goff, gb, gv)
            assert np.array_equal(goff - goff[0], off)
            exact = np.diff(off) != 1
            assert np.array_equal(gb[exact].view(np.uint64), cb[exact].view(np.uint64))
            assert np.array_equal(gv[exact].view(np.uint64), cv[exact].view(np.uint64))
    d.close()
