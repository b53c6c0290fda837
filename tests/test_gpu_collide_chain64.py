"""The FP64 chain kernel (worker warps of 32 swarms, and mass, choice and clock
warps) against the FP64 oracle, event by event, with and without the stored
matrix, at the sizes where its layout changes: single swarms, group edges, the
slot counts of its instantiations (128, 256, 512 swarms).  Masses over fourteen
decades, so that the groups' rates differ by more than 2^57 too.

Both draw the same random numbers and form the rates to a few 1e-16 each (row
sums, kept by updates, to 1e-13 of the total), so a choice differs with a
probability of about n x 1e-13: never here.  Waiting times are held to 1e-11,
and so are masses, whose fragment draws amplify a rounding by up to 1e3.  A lone
swarm takes no ramp: it only meets itself, and every ramped draw, u3 / p of the
mass before, multiplies a rounding by 1.17 on average, 1e16 in 240 events."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
EVENTS = 300


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("store", [0, 2])
@pytest.mark.parametrize("ramp", [0.0, 0.4], ids=["sharp", "ramp"])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 96, 128, 129, 256, 257, 400, 512])
def test_fp64_chain_follows_the_oracle(n, ramp, store):
    if n == 1 and ramp:
        pytest.skip("a chaotic chain")
    P = W.benchmark_disk(v_frag=100.0, frag_ramp=ramp)
    rng = np.random.default_rng(n)
    r, z = 1.3 * W.AU * (1 + rng.uniform(-0.05, 0.05, n)), rng.normal(0, 1, n) * 2e11
    d = mcd.Disk(P, (1, 1, n), seed=17, prec="fp64")
    for key, v in ((mcd.MCD_OPT_DV_MATRIX, store), (mcd.MCD_OPT_LOG_CELL, 0), (mcd.MCD_OPT_CAP_STOPS, 1),
                   (mcd.MCD_OPT_MAX_EVENTS, EVENTS), (mcd.MCD_OPT_REBUILD_EVERY, 97)):
        mcd.mcd_set_option(d.ctx, key, v)
    mcd.mcd_set_particles(d.ctx, 0, W.random_masses(n, seed=n, lo=1e-11, hi=1e3), np.full(n, 2e26), r, z,
                          np.arange(n, dtype=np.uint32))
    mcd.mcd_regrid(d.ctx)
    b, V = np.zeros((1, 6)), np.zeros(1)
    mcd.mcd_get_cells(d.ctx, 0, None, b, V)
    cell = d.particles()
    mcd.mcd_collide(d.ctx, 1e30)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    ijo, t, mnew, nlog = mcd.mcd_get_event_log(d.ctx, 1000)
    st, m_o, ev_o, _, lg = oracle.collide_cell(P, b[0, 4], b[0, 5], V[0], cell["m"], cell["M"], 0.0, 1e30, 17, 0, 0, 0,
                                               max_events=EVENTS, rebuild_every=97, log_cap=1000)
    assert nlog == ev_o == d.stats().events
    assert np.array_equal(ijo[:, 0], lg["i"]) and np.array_equal(ijo[:, 1], lg["j"])
    assert np.array_equal(ijo[:, 2], lg["outcome"])
    assert np.max(np.abs(t / lg["t"] - 1), initial=0) < 1e-11
    assert np.max(np.abs(mnew / lg["m_new"] - 1), initial=0) < 1e-11
    assert np.max(np.abs(d.particles()["m"] / m_o - 1)) < 1e-11
    d.close()
