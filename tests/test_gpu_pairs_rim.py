"""The plain neighbour sums where a term's size and a value's size part: a much larger neighbour near the
kernel's rim (2 - r/h down to 1e-5), components many decades apart, particles on a line.  Every sum keeps
the accuracy of FP64 terms.  Against the same sums in extended precision from the state read back."""
import numpy as np
import pytest

from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _event(dim, delta, line, diffusion=False):
    """A light particle 0, two heavy ones at its rim, a light one close by, one out of reach; scales
    of S 14 decades apart, of u up to 13."""
    ev = (I.smooth_blob_2p1(half_width=0.1, with_table=False, viscous=False) if dim == 2 else
          I.smooth_blob_3d(milne=False, half_widths=(0.16, 0.16, 0.12), with_table=False, viscous=False))
    h = ev.h
    e = np.eye(3) if line else np.array([[0.8, 0.48, 0.36], [-0.59, 0.79, 0.17], [0.1, -0.6, 0.79]])
    e = e[:, :dim]
    e = e / np.sqrt(np.sum(e * e, axis=1, keepdims=True)) if not line else np.stack([e[0], -e[0], e[0]])
    x = np.stack([0.0 * e[0], (2.0 - delta) * h * e[0], (2.0 - 3.0 * delta) * h * e[1], 0.3 * h * e[2], 9.0 * h * e[0]])
    n = len(x)
    ev.x = np.ascontiguousarray(x.T) + 0.3
    ev.S = np.array([1e-13, 1.0, 1e-6, 3e-14, 2.0]) * 0.3
    ev.Nq = np.stack([0.0 * ev.S, 0.01 * ev.S, 0.01 * ev.S])
    ev.Nq[0, 1:] = [0.01, 1e-9, 0.0, 0.0]
    u = np.array([[0.1, -0.2, 0.3], [0.5, 1e-11, -1e-7], [1e-9, -0.3, 1e-3], [1e-13, 1e-14, 0.7e-12], [0.0, 0.0, 0.0]])
    ev.u = np.ascontiguousarray(u[:, :dim].T)
    ev.Bv, ev.Pv = np.zeros(n), np.zeros((3 if dim == 2 else 5, n))
    ev.dtau = 1e-30  # one step sizes the lists without moving the state
    if diffusion:
        ev.diffusion = I.Diffusion(kappaT2=I.KAPPA_BSQ)
    return ev


def _kernel(x, h, dim):
    """w, g (dim) of every pair in extended precision, and the relative error an FP64 evaluation may
    have: the separation's 6 roundings of r/h near 2, three powers of 2 - r/h, 8 more operations."""
    L = np.longdouble
    d = (x.astype(L)[:, :, None] - x.astype(L)[:, None, :])
    r = np.sqrt(np.sum(d * d, axis=0))
    q = r / L(h)
    near = q < 2
    w = np.where(q < 1, 1 - q * q * (L(1.5) - L(0.75) * q), L(0.25) * (2 - q) ** 3)
    dw = np.where(q < 1, -q * (3 - L(2.25) * q), -L(0.75) * (2 - q) ** 2)
    g = np.where(near & (r > 0), dw / np.where(r > 0, r, 1), 0) * d
    tol = EPS * (16 + 36 / np.maximum(2 - q, EPS))
    return np.where(near, w, 0), g, np.where(near, tol, 0), near


@pytest.mark.parametrize("lists", [False, True])
@pytest.mark.parametrize("line", [False, True])
@pytest.mark.parametrize("delta", [0.1, 1e-2, 1e-3, 1e-5])
@pytest.mark.parametrize("dim", [2, 3])
def test_sums_keep_the_accuracy_of_their_terms(dim, delta, line, lists):
    ev = _event(dim, delta, line)
    g = Bd.GpuEvent(ev)
    if lists:
        g.step(1, sync=True)
    st = g.read(("X", "U", "S", "NQ"))
    tau = g.totals()["tau"]
    f = g.read(("NNB", "SIGMA_STAR", "S_DENS", "N_DENS", "P", "STATUS"))
    grad = g.rates()[1]
    g.free()
    L = np.longdouble
    w, gk, tol, near = _kernel(st["X"], ev.h, dim)
    assert np.array_equal(f["NNB"], near.sum(axis=1))
    assert not np.any(f["STATUS"] & ~np.uint32(2))
    sd = (L(10) / (7 * L(np.pi)) if dim == 2 else 1 / L(np.pi)) / L(ev.h) ** dim
    sqrtg = L(tau) if ev.milne else L(1)
    vol = np.sqrt(1 + np.sum(st["U"].astype(L) ** 2, axis=0)) * sqrtg

    def check(got, terms, what):
        """terms [a, b]: each off by its own bound, a rounding per addition, a few after the sum"""
        want, mag = terms.sum(axis=1), np.abs(terms)
        bound = (mag * tol).sum(axis=1) + EPS * (len(terms) + 8) * mag.sum(axis=1)
        assert np.all(np.abs(got - want) <= bound), (what, got, want, bound)

    check(f["SIGMA_STAR"], sd * w, "sigma*")
    check(f["S_DENS"], sd * w * st["S"].astype(L)[None, :] / vol[:, None], "s")
    for k in range(3):
        check(f["N_DENS"][k], sd * w * st["NQ"][k].astype(L)[None, :] / vol[:, None], f"n{k}")
    c = sd / L(ev.h)
    us = st["U"].astype(L) / f["SIGMA_STAR"].astype(L)
    X = f["P"].astype(L) / f["SIGMA_STAR"].astype(L) ** 2  # ideal fluid: X^{ji} = p delta^{ji} / sigma*^2
    for k in range(dim):
        for j in range(dim):
            check(grad[dim * k + j], c * gk[k] * us[j][None, :], f"d_{k} u^{j}")
    for i in range(dim):
        got = grad[dim * dim + i]
        t1, t2 = X[:, None] * gk[i], X[None, :] * gk[i]
        want = -sqrtg * c * (t1.sum(axis=1) + t2.sum(axis=1))
        mag = sqrtg * c * (np.abs(t1) + np.abs(t2))
        bound = (mag * tol).sum(axis=1) + EPS * (len(got) + 12) * mag.sum(axis=1)
        assert np.all(np.abs(got - want) <= bound), (i, got, want, bound)


@pytest.mark.parametrize("line", [False, True])
@pytest.mark.parametrize("delta", [0.1, 1e-3, 1e-5])
def test_diffusion_sums_against_the_cell_pass(delta, line, monkeypatch):
    """Currents after one step with lists against the same step with the FP64 cell pass: J^i_q / sigma of
    a particle is linear in its sums, whose terms agree within both forms' bounds."""
    out = []
    for lists in ("1", "0"):
        monkeypatch.setenv("SPH_PAIR_LISTS", lists)
        ev = _event(2, delta, line, diffusion=True)
        ev.u = 0.0 * ev.u
        g = Bd.GpuEvent(ev)
        g.step(1, sync=True)
        out.append((g.read(("JV",))["JV"], g.read(("SIGMA_STAR", "T", "MU", "P", "X"))))
        g.free()
    (j1, f), (j0, _) = out
    w, gk, tol, near = _kernel(f["X"], ev.h, 2)
    al = (f["MU"] / f["T"]).astype(np.longdouble)
    kap = np.array(I.KAPPA_BSQ)
    for i in range(2):
        for q in range(3):
            # at rest the current starts along sum kappa_{qq'} (alpha_b - alpha_a) grad W of the particle, whose
            # terms carry both forms' kernel bounds and those of the densities behind alpha (T: a cube root;
            # mu/T: n and T)
            terms = sum(kap[q][p] * (al[p][None, :] - al[p][:, None]) * gk[i] for p in range(3))
            err = sum(abs(kap[q][p]) * (np.abs(al[p][None, :]) + np.abs(al[p][:, None])) * np.abs(gk[i]) for p in range(3))
            want = j0[2 * q + i]
            total = np.abs(terms.sum(axis=1))
            factor = np.abs(want) / np.where(total > 0, total, 1)
            bound = factor * (8 * tol.max() * err).sum(axis=1)
            assert np.all(np.abs(j1[2 * q + i] - want) <= bound), (q, i, j1[2 * q + i], want, bound)
