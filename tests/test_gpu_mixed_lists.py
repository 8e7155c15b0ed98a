"""Mixed 3+1D form: the gradient pass over the density pass's neighbour lists adds the same terms in the
same order as the walk (SPH_PAIR_LISTS=0, and the stages whose lists overflow), so the states are
equal bit for bit: one particle, an odd last one, rows past a lane's plain run of sums."""
import numpy as np
import pytest

from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _event(n, extent):
    ev = I.smooth_blob_3d(milne=True, half_widths=(0.16, 0.16, 0.12), with_table=False)
    w = 1.0 + 0.2 * I.uniform01(5, n)
    ev.x, ev.u = I.random_points(n, 3, extent, 61 + n), 0.3 * I.random_points(n, 3, 1.0, 77)
    ev.S, ev.Nq = w, 0.01 * (2.0 * I.uniform01(6, 3 * n).reshape(3, n) - 1.0) * w
    ev.Bv, ev.Pv = np.zeros(n), np.zeros((ev.Pv.shape[0], n))
    return ev


@pytest.mark.parametrize("n,extent", [(1, 0.1), (3, 0.1), (1331, 2.0), (2501, 0.2)])
def test_lists_and_walk_agree(n, extent, monkeypatch):
    def run(**env):
        for k in ("SPH_PAIR_LISTS", "SPH_PAIR_TOTAL", "SPH_PAIR_MARGIN"):
            monkeypatch.delenv(k, raising=False)
        for k, t in env.items():
            monkeypatch.setenv(k, t)
        g = Bd.GpuEvent(_event(n, extent), precision=Bd.SPH_MIXED)
        for _ in range(3):
            g.step(1)
        out = g.read(("X", "U", "S", "BV", "PV", "NNB")), g.totals()
        g.free()
        return out

    a, ta = run()
    assert ta["pair_overflows"] == 0
    for env in ({"SPH_PAIR_LISTS": "0"}, {"SPH_PAIR_TOTAL": "1"}, {"SPH_PAIR_MARGIN": "0"}):
        b, tb = run(**env)
        assert ta["pairs"] == tb["pairs"]
        if env.get("SPH_PAIR_TOTAL"):
            assert tb["pair_overflows"] >= (1 if n > 1 else 0)
        for k in a:
            assert np.array_equal(a[k], b[k], equal_nan=True), (env, k)
