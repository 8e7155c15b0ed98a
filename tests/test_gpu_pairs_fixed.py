"""The plain neighbour sums over pair lists, accumulated in integers, at their edges: one particle, an
odd last particle, cells of a few particles, coincident particles, values over many decades between
neighbours, zeros, and more neighbours than the accumulators hold without folding."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# sums of terms that carry a few ulp each: against the oracle's FP64 sums of up to 2,500 terms
TOL = 1e-13


def _event(dim, n, extent, decades, coincident):
    if dim == 2:
        ev = I.smooth_blob_2p1(half_width=0.1, with_table=False)
    else:
        ev = I.smooth_blob_3d(milne=False, half_widths=(0.16, 0.16, 0.12), with_table=False)
    x = I.random_points(n, dim, extent, 50 + n)
    if coincident:
        x[:, 1::2] = x[:, 0:n - 1:2]
    w = 10.0 ** (decades * (I.uniform01(8, n) - 0.5))
    ev.x, ev.u = x, 0.3 * I.random_points(n, dim, 1.0, 78)
    ev.S, ev.Nq = w, 0.01 * (2.0 * I.uniform01(9, 3 * n).reshape(3, n) - 1.0) * w
    ev.Nq[1, ::3] = 0.0
    ev.Bv, ev.Pv = np.zeros(n), np.zeros((3 if dim == 2 else 5, n))
    return ev


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n,extent,decades,coincident", [(1, 0.1, 0.0, False), (2, 0.2, 6.0, False), (3, 3.0, 0.0, False),
                                                         (67, 1.0, 3.0, False), (64, 0.5, 0.0, True),
                                                         (501, 0.8, 8.0, False), (2501, 0.17, 1.0, False)])
def test_fixed_sums_against_oracle(dim, n, extent, decades, coincident):
    ev = _event(dim, n, extent, decades, coincident)
    g = Bd.GpuEvent(ev)
    g.step(1, sync=True)  # sizes the lists; the state then differs from the initial one
    st = g.read(("X", "U", "S", "BV", "PV", "GUESS"))
    tau = g.totals()["tau"]
    f = g.read(("NNB", "SIGMA_STAR", "S_DENS", "N_DENS"))
    rates, grad = g.rates()
    run = O.OracleRun.start(ev)
    run.step(1)
    run.y = np.concatenate([st["X"], st["U"], st["S"][None], st["BV"][None], st["PV"]])
    run.tau, run.guess = tau, st["GUESS"]
    aux, _ = run.observe()
    A = O.AUX
    assert np.array_equal(f["NNB"], aux[A["nnb"]].astype(np.int32))
    # pointwise where all terms have one sign
    assert np.max(np.abs(f["SIGMA_STAR"] / aux[A["sigstar"]] - 1.0)) < TOL
    assert np.max(np.abs(f["S_DENS"] / aux[A["s"]] - 1.0)) < TOL
    # charges: against the sum of the terms' magnitudes (|N| <= 0.01 S)
    assert np.max(np.abs(f["N_DENS"] - aux[A["nB"]:A["nQ"] + 1]) / aux[A["s"]]) < 0.01 * TOL
    og = run.stage()[2]
    for rows in (slice(0, dim * dim), slice(dim * dim, dim * dim + dim)):
        assert np.max(np.abs(grad[rows] - og[rows])) <= 10 * TOL * max(np.max(np.abs(og[rows])), 1e-300)
    g.free()


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n,extent,decades,coincident", [(1, 0.1, 0.0, False), (3, 3.0, 0.0, False), (64, 0.5, 0.0, True),
                                                         (501, 0.8, 8.0, False), (2501, 0.17, 1.0, False)])
def test_densities_without_lists_against_oracle(dim, n, extent, decades, coincident):
    """A new state's read-out (no lists yet): the per-particle density pass."""
    ev = _event(dim, n, extent, decades, coincident)
    g = Bd.GpuEvent(ev)
    f = g.read(("NNB", "SIGMA_STAR", "S_DENS", "N_DENS"))
    aux, _ = O.OracleRun.start(ev).observe()
    A = O.AUX
    assert np.array_equal(f["NNB"], aux[A["nnb"]].astype(np.int32))
    assert np.max(np.abs(f["SIGMA_STAR"] / aux[A["sigstar"]] - 1.0)) < TOL
    assert np.max(np.abs(f["S_DENS"] / aux[A["s"]] - 1.0)) < TOL
    assert np.max(np.abs(f["N_DENS"] - aux[A["nB"]:A["nQ"] + 1]) / aux[A["s"]]) < 0.01 * TOL
    g.free()
