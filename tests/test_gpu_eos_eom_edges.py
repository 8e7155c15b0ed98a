"""The EoS search and finish kernels over the whole range of densities (below, inside, at the edges of
and above the table; cold and warm starts; block remainders), and the minimal Israel-Stewart equations
of motion at random viscous states, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-11  # the plain form's bar for one stage (tests/test_gpu_parity.py)


def _lone_particles(n, table, eos, chi_off=False):
    """n particles out of each other's reach: the densities are S W(0), chosen over 10 decades."""
    ev = I.smooth_blob_2p1(half_width=0.1, with_table=False, eos=eos)
    k = int(np.ceil(np.sqrt(n)))
    g = np.arange(n)
    ev.x = np.stack([2.0 * (g % k), 2.0 * (g // k)]).astype(float)
    w0 = 10.0 / (7.0 * np.pi * ev.h ** 2)
    s = 10.0 ** (-5.0 + 10.0 * I.uniform01(3, n))
    ev.S = s * ev.tau0 / w0
    r = 0.0 if chi_off else 0.03
    ev.Nq = r * (2.0 * I.uniform01(4, 3 * n).reshape(3, n) - 1.0) * ev.S
    ev.u, ev.Bv, ev.Pv = np.zeros((2, n)), np.zeros(n), np.zeros((3, n))
    ev.table = table
    return ev


@pytest.mark.parametrize("form", ["table", "closed", "conformal"])
@pytest.mark.parametrize("n", [1, 63, 65, 1500])
def test_eos_over_the_density_range(form, n):
    eos = I.AnalyticEoS(a0=11.0 / 3.0) if form == "conformal" else I.BJ_EOS
    table = I.synthetic_eos_table(I.BJ_EOS, nT=64, nmu=16) if form == "table" else None
    ev = _lone_particles(n, table, eos, chi_off=form == "conformal")
    g = Bd.GpuEvent(ev)
    run = O.OracleRun.start(ev)
    A = O.AUX
    for steps in (0, 1, 2):  # cold, then from the warm starts
        if steps:
            g.step(1, sync=True)
            run.step(1)
        f = g.read(("T", "MU", "P", "E", "STATUS"))
        aux, st = run.observe()
        assert np.array_equal(f["STATUS"], st)
        for k, v in (("T", aux[A["T"]]), ("P", aux[A["p"]]), ("E", aux[A["e"]])):
            assert np.max(np.abs(f[k] - v) / np.maximum(np.abs(v), 1e-300)) < 1e-10, k
            assert np.max(np.abs(f[k] - v)) <= TOL * np.max(np.abs(v)), k
        mu = aux[A["muB"]:A["muQ"] + 1]
        assert np.max(np.abs(f["MU"] - mu)) <= TOL * max(np.max(np.abs(mu)), 1e-300)
    g.free()


@pytest.mark.parametrize("dim,milne", [(2, True), (2, False), (3, True), (3, False)])
@pytest.mark.parametrize("n", [1, 64, 321])
def test_rates_of_random_viscous_states(dim, milne, n):
    if dim == 2:
        ev = I.smooth_blob_2p1(half_width=0.1, with_table=False, eos=I.CAUSAL_EOS)
        ev.milne = milne
    else:
        ev = I.smooth_blob_3d(milne=milne, half_widths=(0.16, 0.16, 0.12), with_table=False, eos=I.CAUSAL_EOS)
    npi = 3 if dim == 2 else 5
    ev.x = I.random_points(n, dim, 0.5, 41)
    ev.u = I.random_points(n, dim, 0.8, 42)
    ev.S = 0.05 + 0.1 * I.uniform01(43, n)
    ev.Nq = 0.02 * (2.0 * I.uniform01(44, 3 * n).reshape(3, n) - 1.0) * ev.S
    ev.Bv = 0.02 * (2.0 * I.uniform01(45, n) - 1.0)
    ev.Pv = 0.02 * (2.0 * I.uniform01(46, npi * n).reshape(npi, n) - 1.0)
    g = Bd.GpuEvent(ev)
    rates, _ = g.rates()
    want = O.OracleRun.start(ev).stage()[0]
    for k in range(want.shape[0]):
        assert np.max(np.abs(rates[k] - want[k])) <= TOL * max(np.max(np.abs(want[k])), 1e-300), k
    g.free()
