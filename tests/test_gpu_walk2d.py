"""The mixed 2+1D neighbour walk at its edges: one particle, an odd last particle, two particles of a
warp in different cells, coincident particles, and more neighbours than a lane sums in plain FP32."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the mixed form's bar (see test_gpu_walk3d.py)


@pytest.mark.parametrize("n,extent,coincident", [(1, 0.1, False), (2, 3.0, False), (3, 0.2, False), (67, 1.0, False),
                                                 (901, 3.0, False), (64, 0.5, True), (2501, 0.2, False)])
def test_mixed_walk_against_oracle(n, extent, coincident):
    ev = I.smooth_blob_2p1(half_width=0.1, with_table=False)
    x = I.random_points(n, 2, extent, 61 + n)
    if coincident:
        x[:, 1::2] = x[:, 0:n - 1:2]
    w = 1.0 + 0.2 * I.uniform01(5, n)
    ev.x, ev.u = x, 0.3 * I.random_points(n, 2, 1.0, 77)
    ev.S, ev.Nq = w, 0.01 * (2.0 * I.uniform01(6, 3 * n).reshape(3, n) - 1.0) * w
    ev.Bv, ev.Pv = np.zeros(n), np.zeros((3, n))
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
    for rows in (slice(0, 4), slice(4, 6)):
        assert np.max(np.abs(grad[rows] - og[rows])) <= TOL * max(np.max(np.abs(og[rows])), 1e-300)
    g.free()
