"""The mixed chain kernel's first row sums and first look at the clock.

The row sums come from a stored matrix (each pair once, spread over all threads), or
without one from the owners' fresh entries and from columns that the warps without
swarms form: the same bits whatever the store, the thread count and the memory left
for columns.  (The total rate's bits depend on the thread count: the groups' totals
are added in a tree over the thread count's groups.)  A cell whose first waiting time lies beyond t_end ends there: its
events, masses, row sums and total rate are those of the whole chain (oracle:
events exactly, rates to the mixed path's 1e-5)."""
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


def _cells(n, cells, opts):
    """(context, columns, bounds, volumes) of a row of cells with random masses."""
    P = W.benchmark_disk(v_frag=100.0)
    d = mcd.Disk(P, (cells, 1, n), seed=17, prec="mixed")
    for key, v in ((mcd.MCD_OPT_SWARMS_PER_THREAD, 1), (mcd.MCD_OPT_DUMP_R, 1), *opts):
        mcd.mcd_set_option(d.ctx, key, v)
    N = n * cells
    rng = np.random.default_rng(n)
    r, z = W.AU * (1 + 2 * rng.random(N)), rng.normal(0, 1, N) * 2e11
    mcd.mcd_set_particles(d.ctx, 0, W.random_masses(N, seed=n, lo=1e-8, hi=1e2), np.full(N, 2e26), r, z,
                          np.arange(N, dtype=np.uint32))
    mcd.mcd_regrid(d.ctx)
    b, V = np.zeros((cells, 6)), np.zeros(cells)
    mcd.mcd_get_cells(d.ctx, 0, None, b, V)
    return P, d, d.particles(), b, V


def _rates(d, N, cells):
    R, Rtot = np.zeros(N), np.zeros(cells)
    mcd.mcd_get_rates(d.ctx, 0, R)
    mcd.mcd_get_total_rates(d.ctx, 0, Rtot)
    return R, Rtot


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 31, 32, 33, 63, 64, 65, 97, 128, 223, 256, 290, 300, 318, 319, 401, 480, 512])
def test_row_sums_have_the_same_bits_however_they_are_built(n):
    ref, total = None, {}
    shapes = [(store, o) for store in (0, 1, 2) for o in ([], [(mcd.MCD_OPT_EXCLUSIVE, 0)], [(mcd.MCD_OPT_THREADS, 512)])]
    for store, o in shapes:
        _, d, x, _, _ = _cells(n, 3, [(mcd.MCD_OPT_DV_MATRIX, store), (mcd.MCD_OPT_CAP_STOPS, 1),
                                      (mcd.MCD_OPT_MAX_EVENTS, 0), *o])
        mcd.mcd_collide(d.ctx, 1e30)
        assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
        got = _rates(d, 3 * n, 3)
        d.close()
        if ref is None:
            ref = got
            assert np.all(got[0] > 0) and np.all(got[1] > 0)
        threads = o[0][1] if o and o[0][0] == mcd.MCD_OPT_THREADS else 0
        assert np.array_equal(got[0], ref[0]), (store, o)
        assert np.array_equal(got[1], total.setdefault(threads, got[1])), (store, o)


@pytest.mark.parametrize("store", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 8, 32, 33, 64, 65, 200, 300, 400])
def test_cells_without_an_event_match_the_oracle(n, store):
    cells = 24
    P, d, x, b, V = _cells(n, cells, [(mcd.MCD_OPT_DV_MATRIX, store)])
    total = np.array([oracle.rate_matrix(P, b[c, 4], b[c, 5], V[c], x["m"][c * n:c * n + n], x["M"][c * n:c * n + n])[1].sum()
                      for c in range(cells)])
    t_end = 0.7 / np.median(total)
    mcd.mcd_collide(d.ctx, t_end)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    ev = np.zeros(cells, np.int64)
    mcd.mcd_get_cell_events(d.ctx, 0, ev)
    got = d.particles()
    R, Rtot = _rates(d, n * cells, cells)
    d.close()
    none = 0
    for c in range(cells):
        s = slice(c * n, c * n + n)
        _, m_o, ev_o, _, _ = oracle.collide_cell(P, b[c, 4], b[c, 5], V[c], x["m"][s], x["M"][s], 0.0, t_end, 17, 0, 0, c)
        assert ev[c] == ev_o
        assert np.max(np.abs(got["m"][s] / m_o - 1)) < 2e-5
        R_o = oracle.rate_matrix(P, b[c, 4], b[c, 5], V[c], got["m"][s], got["M"][s])[1]
        assert np.max(np.abs(R[s] / R_o - 1)) < 1e-5
        if ev_o == 0:
            none += 1
            assert np.array_equal(got["m"][s], x["m"][s]) and abs(Rtot[c] / R_o.sum() - 1) < 1e-5
    assert none >= 3 and none < cells
