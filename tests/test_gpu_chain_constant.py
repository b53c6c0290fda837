"""The mixed chain kernel with the constant kernel (a branch of its own in the pair
entries and the swarm caches) against the oracle, event by event, with and without
grouping.  Masses add exactly; 40 choices differ by FP32 roundings with a
probability below 1e-2 at 512 swarms; waiting times hold to 2e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
EVENTS = 40


@pytest.mark.parametrize("dm", [0.0, 0.3])
@pytest.mark.parametrize("store", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 33, 64, 200, 318, 319, 512])
def test_constant_kernel_chain_follows_the_oracle(n, store, dm):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()
    P = W.constant_kernel_cell(dm_group=dm)
    rng = np.random.default_rng(n)
    m = rng.integers(1, 20, n).astype(float)
    d = mcd.Disk(P, (1, 1, n), seed=17, prec="mixed")
    for key, v in ((mcd.MCD_OPT_SWARMS_PER_THREAD, 1), (mcd.MCD_OPT_DV_MATRIX, store), (mcd.MCD_OPT_LOG_CELL, 0),
                   (mcd.MCD_OPT_CAP_STOPS, 1), (mcd.MCD_OPT_MAX_EVENTS, EVENTS), (mcd.MCD_OPT_REBUILD_EVERY, 23)):
        mcd.mcd_set_option(d.ctx, key, v)
    mcd.mcd_set_particles(d.ctx, 0, m, np.full(n, 1.0 / n), W.AU * (1 + rng.random(n)), rng.normal(0, 1, n),
                          np.arange(n, dtype=np.uint32))
    mcd.mcd_regrid(d.ctx)
    cell = d.particles()
    mcd.mcd_collide(d.ctx, 1e30)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    ijo, t, mnew, nlog = mcd.mcd_get_event_log(d.ctx, 1000)
    _, m_o, ev_o, _, lg = oracle.collide_cell(P, 1.5 * W.AU, 0.0, 1.0, cell["m"], cell["M"], 0.0, 1e30, 17, 0, 0, 0,
                                              max_events=EVENTS, rebuild_every=23, log_cap=1000)
    assert nlog == ev_o == EVENTS
    assert np.array_equal(ijo[:, 0], lg["i"]) and np.array_equal(ijo[:, 1], lg["j"])
    assert np.max(np.abs(t / lg["t"] - 1)) < 2e-5
    assert np.max(np.abs(d.particles()["m"] / m_o - 1)) < 1e-15
    d.close()
