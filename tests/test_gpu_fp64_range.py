"""The FP64 path's reciprocals at the edges of the FP32 range they start from.

1/m, 1/(dm m), 1/(1 + St^2) and L/R_tot take a reciprocal seeded by the FP32
special-function unit for operands it can represent and the plain division for
the others; above 2^126 the FP32 reciprocal is subnormal and flushed to zero.
The constant kernel has free units, so masses and total rates at 2^-75, 2^-74 and
from 2^125 to 2^128 are legal; pairs of bodies with Stokes numbers around 2^63
reach the range through 1 + St^2.  Each against the oracle: the same events,
times, masses and kernel entries to 1e-12 (a dozen roundings of 1.1e-16, and what
FP64 itself leaves of 1 - St_i St_j)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2507_21239_gb300 import mcd, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
EVENTS, N = 40, 33
EDGES = [2.0**-75, 2.0**-74, 2.0**125, 1.5 * 2.0**125, 2.0**126 * (1 - 2.0**-53), 2.0**126 * (1 + 2.0**-52),
         1.5 * 2.0**126, 2.0**127 * (1 - 2.0**-53), 2.0**127, 1.5 * 2.0**127]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21239_gb300 import build
    build.build()
    oracle.build()


def _follows_the_oracle(P, m, M):
    d = mcd.Disk(P, (1, 1, m.size), seed=17, prec="fp64")
    for key, v in ((mcd.MCD_OPT_LOG_CELL, 0), (mcd.MCD_OPT_CAP_STOPS, 1), (mcd.MCD_OPT_MAX_EVENTS, EVENTS)):
        mcd.mcd_set_option(d.ctx, key, v)
    rng = np.random.default_rng(3)
    mcd.mcd_set_particles(d.ctx, 0, m, M, W.AU * (1 + rng.random(m.size)), rng.normal(0, 1, m.size) * 2e11,
                          np.arange(m.size, dtype=np.uint32))
    mcd.mcd_regrid(d.ctx)
    cell = d.particles()
    mcd.mcd_collide(d.ctx, 1e60)
    assert mcd.mcd_sync(d.ctx) == mcd.MCD_OK
    ijo, t, mnew, nlog = mcd.mcd_get_event_log(d.ctx, 1000)
    _, m_o, ev_o, _, lg = oracle.collide_cell(P, 1.5 * W.AU, 0.0, 1.0, cell["m"], cell["M"], 0.0, 1e60, 17, 0, 0, 0,
                                              max_events=EVENTS, log_cap=1000)
    assert nlog == ev_o == EVENTS
    assert np.array_equal(ijo[:, 0], lg["i"]) and np.array_equal(ijo[:, 1], lg["j"])
    assert np.max(np.abs(t / lg["t"] - 1)) < 1e-12
    assert np.max(np.abs(mnew / lg["m_new"] - 1)) < 1e-12
    assert np.max(np.abs(d.particles()["m"] / m_o - 1)) < 1e-12
    d.close()


@pytest.mark.parametrize("edge", EDGES, ids=lambda x: f"2^{np.log2(x):.2f}")
@pytest.mark.parametrize("dm", [0.0, 1e-3])
def test_masses_at_the_range_edges(edge, dm):
    """Masses (dm = 0) or group masses dm m (dm > 0) at the edge."""
    P = W.constant_kernel_cell(dm_group=dm)
    rng = np.random.default_rng(5)
    m = edge / (dm if dm else 1.0) * np.where(rng.random(N) < 0.5, 1.0, 1.0 + 0.4 * rng.random(N))
    _follows_the_oracle(P, m, m / N)


@pytest.mark.parametrize("edge", EDGES, ids=lambda x: f"2^{np.log2(x):.2f}")
def test_total_rates_at_the_range_edges(edge):
    m = np.full(N, 2.0)
    P = W.constant_kernel_cell(K_const=edge / (N * 0.5))  # R_tot = N sum_j K (M_j / m_j) = N K / 2
    _follows_the_oracle(P, m, np.full(N, 1.0 / N))


def test_stokes_numbers_at_the_range_edge():
    P = W.benchmark_disk()
    rc, zc = 2.0 * W.AU, 1e11
    m = np.geomspace(1e-12, 1e60, 4000)
    _, St, _ = oracle.particle(P, rc, zc, m)
    mi = m[(St > 2.0**61) & (St < 2.0**66)]
    assert mi.size > 50 and St.max() > 2.0**66
    mi, mj = np.concatenate([mi, mi, mi]), np.concatenate([2.0 * mi, np.full(mi.size, 1e-3), mi[::-1]])
    ref = oracle.pairs(P, rc, zc, mi, mj)
    ti, tj = torch.tensor(mi, device="cuda"), torch.tensor(mj, device="cuda")
    dv, K = torch.empty_like(ti), torch.empty_like(ti)
    mcd.mcd_pair_probe(P, mcd.MCD_FP64, rc, zc, ti, tj, dv, K)
    torch.cuda.synchronize()
    assert np.all(np.abs(dv.cpu().numpy() - ref["dv"]) <= 1e-12 * ref["dv"])
    assert np.all(np.abs(K.cpu().numpy() - ref["K"]) <= 1e-12 * ref["K"])
