"""The mixed 3+1D neighbour walk at its edges: one particle, an odd last particle, two particles
of a warp in different cells, cells of a few particles, coincident particles, and more neighbours
than a lane sums in plain FP32 (1,024)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# per-lane runs of at most 32 plain terms (32 * 2^-24 = 1.9e-6 of the terms' magnitudes) and kernel
# values good to a few 2^-22: the mixed form's bar
TOL = 1e-5


def _event(n, extent, coincident):
    ev = I.smooth_blob_3d(milne=False, half_widths=(0.16, 0.16, 0.12), with_table=False)
    x = I.random_points(n, 3, extent, 31 + n)
    if coincident:
        x[:, 1::2] = x[:, 0:n - 1:2]
    w = 1.0 + 0.2 * I.uniform01(5, n)
    ev.x, ev.u = x, 0.3 * I.random_points(n, 3, 1.0, 77)
    ev.S, ev.Nq = w, 0.01 * (2.0 * I.uniform01(6, 3 * n).reshape(3, n) - 1.0) * w
    ev.Bv, ev.Pv = np.zeros(n), np.zeros((5, n))
    return ev


@pytest.mark.parametrize("n,extent,coincident", [(1, 0.1, False), (2, 3.0, False), (3, 0.2, False), (67, 1.0, False),
                                                 (501, 1.5, False), (64, 0.5, True), (2501, 0.17, False)])
def test_mixed_walk_against_oracle(n, extent, coincident):
    ev = _event(n, extent, coincident)
    g = Bd.GpuEvent(ev, precision=Bd.SPH_MIXED)
    f = g.read(("NNB", "SIGMA_STAR", "S_DENS", "N_DENS"))
    _, grad = g.rates()
    run = O.OracleRun.start(ev)
    aux, _ = run.observe()
    A = O.AUX
    assert np.array_equal(f["NNB"], aux[A["nnb"]].astype(np.int32))
    assert np.max(np.abs(f["SIGMA_STAR"] / aux[A["sigstar"]] - 1.0)) < TOL
    assert np.max(np.abs(f["S_DENS"] / aux[A["s"]] - 1.0)) < TOL
    assert np.max(np.abs(f["N_DENS"] - aux[A["nB"]:A["nQ"] + 1])) < TOL * 0.01 * np.max(aux[A["s"]])
    og = run.stage()[2]
    for rows in (slice(0, 9), slice(9, 12)):
        assert np.max(np.abs(grad[rows] - og[rows])) <= TOL * max(np.max(np.abs(og[rows])), 1e-300)
    g.free()
