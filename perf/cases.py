"""What the SPH framework is timed on: the calls that a program evolving heavy-ion events makes.

Every case goes through the binding of the C ABI, as a user's program does: single events in the
plain FP64 and the mixed form, 2+1D and 3+1D, with the options used in earnest (viscosity, BSQ
charges and diffusion, jets, conformal and tabulated equation of state), an event from its creation to
its end, a read-out of derived fields, and the serving form.  Sizes are those of the repository's
configurations: 2,601 particles (the Gubser lattice), 5 k to 200 k (the serving stream), 40 k (the
benchmark event), about 10^4 to 8 10^6 in 3+1D.

A pass of an event case advances the event and copies its state to device buffers that the program
keeps; the next pass goes on from there, as the event's time loop does (an event at its end starts
again).  The mixed and serving forms carry about single precision (1e-7, include/sph_gb300.h), and
their snapshots are kept as float32; those of the plain form as float64.
"""
import copy
import math

import numpy as np
import torch

from paper_2511_22852_gb300 import binding as Bd
from paper_2511_22852_gb300 import inputs as I

STATE = ("X", "U", "S", "NQ", "BV", "PV", "GUESS")
DERIVED = ("SIGMA_STAR", "S_DENS", "N_DENS", "T", "MU", "P", "E", "STATUS", "NNB")
SERVED = ("X", "U", "S", "BV", "PV", "T", "NNB")
NAMES = {"X": "x", "U": "u", "S": "S", "NQ": "Nq", "BV": "Bv", "PV": "Pv", "GUESS": "guess", "JV": "Jv",
         "SIGMA_STAR": "sigstar", "S_DENS": "s", "N_DENS": "nq", "T": "T", "MU": "mu", "P": "p", "E": "e",
         "STATUS": "status", "NNB": "nnb"}
WORDS = ("STATUS", "NNB")
TABLE = (64, 32)  # nodes along T and along each chemical potential


def listed():
    def ev(name, kind, n, precision="fp64", steps=1, **more):
        return {"name": name, "kind": kind, "n": n, "precision": precision, "steps": steps, **more}

    return [
        # the smallest: a validation run of the ideal Gubser lattice, from creation to its last step
        ev("gubser_2d_whole_run", "gubser", 2601, steps=60),
        # one small event of the stream, alone on the GPU: launches and latency
        ev("bsq_2d_5k_fp64", "bsq2", 5000, steps=8),
        # the benchmark event, in both precisions
        ev("bsq_2d_40k_fp64", "bsq2", 40000, steps=4),
        ev("bsq_2d_40k_mixed", "bsq2", 40000, "mixed", steps=8),
        # the largest 2+1D system of the stream
        ev("bsq_2d_200k_fp64", "bsq2", 200000),
        # BSQ diffusion with the full kappa matrix
        ev("diffusion_2d_21k_fp64", "diff2", 21013, steps=2),
        # densities, temperature and potentials of a new state: initial conditions looked over, snapshots analysed
        ev("observe_2d_40k_fp64", "observe2", 39001),
        # a small 3+1D Cartesian event
        ev("blob_3d_9k_fp64", "blob3", 9261, steps=4),
        # the 3+1D Milne event in both precisions (the mixed one a smaller system at the same resolution)
        ev("milne_3d_1m_fp64", "bsq3", 1012121),
        ev("milne_3d_258k_mixed", "bsq3", 258000, "mixed"),
        # the largest: the 3+1D Cartesian stress event with jets
        ev("stress_3d_8m_mixed", "stress3", 8000000, "mixed"),
        # event-by-event production: eight events of the stream submitted, evolved together and collected
        {"name": "serve_8_events", "kind": "serve", "events": 8, "smallest": 5000, "largest": 200000, "steps": 16},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["gubser", "bsq2", "bsq2", "bsq2", "diff2", "observe2", "blob3", "bsq3", "bsq3", "stress3", "serve"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "gubser":
        return {"kind": kind, "n": rng.randrange(31, 92, 2) ** 2, "precision": "fp64", "steps": rng.randrange(20, 61)}
    if kind == "serve":
        lo = size(5000, 20000)
        return {"kind": kind, "events": rng.randrange(2, 9), "smallest": lo, "largest": size(2 * lo, 200000),
                "steps": rng.randrange(4, 17)}
    if kind in ("bsq2", "diff2", "observe2"):
        n = size(5000, 200000) if kind == "bsq2" else size(5000, 60000)
        return {"kind": kind, "n": n, "precision": precision if kind == "bsq2" else "fp64",
                "steps": 1 if kind == "observe2" else max(1, min(8, 80000 // n))}
    if kind == "blob3":
        return {"kind": kind, "n": rng.randrange(15, 34, 2) ** 3, "precision": precision, "steps": rng.randrange(1, 5)}
    if kind == "bsq3":
        return {"kind": kind, "n": size(60000, 1000000), "precision": precision, "steps": 1}
    return {"kind": kind, "n": size(200000, 3000000), "precision": "mixed", "steps": 1}


# ---------------------------------------------------------------------------
# inputs
def _seeds(seed):
    """Seeds of an event's hotspots and charges, far from those of other seeds."""
    return 1000 + 7919 * int(seed), 500000 + 104729 * int(seed)


def _bsq2(n, seed, tau_end=8.0, T_stop=0.0):
    """The 2+1D viscous BSQ event of about n particles: 200 hotspots per 40,000 particles on a disc
    of 7 fm sqrt(n / 40000), as the serving stream's events."""
    R, hot, q = 7.0 * math.sqrt(n / 40000.0), max(1, round(200 * n / 40000.0)), _seeds(seed)
    e = I.viscous_bsq_2p1(n_target=n, R=R, n_hot=1, seed_charge=q[1], with_table=False, tau_end=tau_end)
    # the hotspots' entropy in place of the single one's (the sum over hotspots taken on the GPU)
    u = I.uniform01(q[0], 2 * hot)
    c = np.stack([R * np.sqrt(u[:hot]) * np.cos(2 * math.pi * u[hot:]), R * np.sqrt(u[:hot]) * np.sin(2 * math.pi * u[hot:])])
    x, c = torch.from_numpy(e.x).cuda(), torch.from_numpy(c).cuda()
    s = torch.zeros_like(x[0])
    for k in range(0, hot, 64):
        s += torch.exp(-((x[0][:, None] - c[0, k:k + 64]) ** 2 + (x[1][:, None] - c[1, k:k + 64]) ** 2) / 0.32).sum(1)
    s = (s * (float(e.S.max()) / float(s.max()))).cpu().numpy()
    e.Nq, e.S = 0.1 * (2.0 * I.uniform01(q[1], 3 * s.size).reshape(3, -1) - 1.0) * s, s
    e.transport = copy.copy(e.transport)
    e.transport.T_stop_GeV = T_stop
    return e


def _event(case, seed):
    kind, n, q = case["kind"], case["n"], _seeds(seed)
    if kind == "gubser":  # the lattice spacing of the 51 x 51 run, its temperature field moved a little by the seed
        e = I.gubser_ideal_2p1(n_side=math.isqrt(n), half_width=0.1 * (math.isqrt(n) - 1), nsteps=case["steps"])
        e.S *= 1.0 + 0.05 * np.sin(1.0 + 0.37 * (seed % 1009) + e.x[0]) * np.cos(e.x[1])
        return e
    if kind in ("bsq2", "observe2"):
        return _bsq2(n, seed)
    if kind == "diff2":
        e = _bsq2(n, seed)
        e.diffusion = I.Diffusion(kappaT2=I.KAPPA_BSQ)
        return e
    if kind == "blob3":
        half = (round(n ** (1.0 / 3.0)) - 1) / 2.0
        e = I.smooth_blob_3d(milne=False, half_widths=(0.16 * half, 0.16 * half, 0.12 * half), flow=0.2, with_table=False,
                             seed_charge=q[1])
        e.S, e.Nq = e.S * (1.0 + 0.1 * np.cos(2.0 * e.x[0] + seed % 1013)), e.Nq
        return e
    if kind == "bsq3":  # the resolution of the 10^6-particle event on a disc of matching radius
        R = 7.0 * math.sqrt(n / 1012121.0)
        return I.viscous_bsq_3p1(R=R, n_hot=max(1, round(200 * n / 1012121.0)), seed_hot=q[0], seed_charge=q[1], with_table=False)
    # the stress event's h over spacing (about 600 neighbours) at every size
    return I.stress_cartesian_3d(n_target=n, h=0.15 * (8.0e6 / n) ** (1.0 / 3.0), seed_hot=q[0], seed_charge=q[1],
                                 seed_tracks=5 + int(seed) % 1000, with_table=False)


_tables, _eos = {}, {}


def _table(shape):
    """The tabulated equation of state, which a program reads once."""
    if shape not in _tables:
        _tables[shape] = I.synthetic_eos_table(I.BJ_EOS, nT=shape[0], nmu=shape[1])
    return _tables[shape]


def _handle(e, shape):
    """The EoS handle: a program makes one and keeps it for all of its events."""
    key = "conformal" if e.eos.a1 == 0.0 else "table %d %d" % shape
    if key not in _eos:
        d, keep = Bd.eos_desc(e.eos, None if key == "conformal" else _table(shape))
        _eos[key] = (Bd.sph_set_eos_table(d), keep if key == "conformal" else None)
    return _eos[key][0]


def _shape(case):
    return (128, 64) if case["kind"] == "stress3" else TABLE


def _gpu_event(case, e):
    return Bd.GpuEvent(e, eos_handle=_handle(e, _shape(case)),
                       precision=Bd.SPH_MIXED if case["precision"] == "mixed" else Bd.SPH_FP64)


def _buffers(e, names):
    """Device buffers of the fields `names` of an event, and the descriptor that hands them over."""
    rows = {"X": e.dim, "U": e.dim, "NQ": 3, "PV": 3 if e.dim == 2 else 5, "GUESS": 4, "JV": 6, "N_DENS": 3, "MU": 3}
    b, out, mask = Bd.FieldBufs(), {}, 0
    b.on_device = 1
    for k in names:
        out[k] = torch.zeros((rows.get(k, 1), e.n), dtype=torch.int32 if k in WORDS else torch.float64, device="cuda")
        setattr(b, NAMES[k], out[k].data_ptr())
        mask |= Bd.F[k]
    return b, out, mask


def prepare(case, seed):
    if case["kind"] == "serve":
        lo, hi = math.log(case["smallest"]), math.log(case["largest"])
        # sizes spread evenly over the logarithm, as the stream's are on average
        sizes = [math.exp(lo + (hi - lo) * (k + 0.5) / case["events"]) for k in range(case["events"])]
        # the stream's stop temperature of 0.10 GeV
        events = [_bsq2(int(n), 100 * int(seed) + k, T_stop=0.10) for k, n in enumerate(sizes)]
        for e in events:
            e.table = None
        table = _table(TABLE)
        need = sum(256 * -(-e.n // 256) for e in events)
        srv = Bd.GpuServer(events[0].eos, table, max_events=case["events"], max_particles=need + 256 * len(events))
        return {"case": case, "server": srv, "events": events}
    e = _event(case, seed)
    if case["kind"] == "gubser":
        return {"case": case, "event": e, "handle": _handle(e, TABLE)}
    names = STATE + (("JV",) if case["kind"] == "diff2" else ())
    if case["kind"] == "observe2":
        first, _, first_mask = _buffers(e, ("X", "U", "S", "BV", "PV"))
        keep = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in
                (("X", e.x), ("U", e.u), ("S", e.S), ("BV", e.Bv), ("PV", e.Pv))}
        for k, v in keep.items():
            setattr(first, NAMES[k], v.data_ptr())
        return {"case": case, "gpu": _gpu_event(case, e), "in": (first, first_mask, keep), "out": _buffers(e, DERIVED)}
    return {"case": case, "event": e, "gpu": _gpu_event(case, e), "out": _buffers(e, names), "done": 0}


def run(state):
    case = state["case"]
    if case["kind"] == "serve":  # submit, evolve together, collect into host arrays
        srv = state["server"]
        tickets = [srv.submit(e, case["steps"]) for e in state["events"]]
        srv.drain()
        got = []
        for t in tickets:
            o = srv.collect(t, SERVED)
            got.append({k: o[k] if k in WORDS else o[k].astype(np.float32) for k in SERVED})
        return got
    if case["kind"] == "gubser":  # an event's whole life
        g = _gpu_event(case, state["event"])
        g.step(case["steps"])
        out = g.read(("X", "U", "S", "T", "E"))
        g.free()
        return out
    b, out, mask = state["out"]
    if case["kind"] == "observe2":
        Bd.sph_write_state(state["gpu"].h, state["in"][1], state["in"][0])
        Bd.sph_read_fields(state["gpu"].h, mask, b, None)
        return out
    if state["done"] + case["steps"] > state["event"].nsteps and state["done"] and case["kind"] in ("bsq2", "diff2"):
        state["gpu"].free()
        state["gpu"], state["done"] = _gpu_event(case, state["event"]), 0
    state["gpu"].step(case["steps"])
    state["done"] += case["steps"]
    Bd.sph_read_fields(state["gpu"].h, mask, b, None)
    if case["precision"] == "mixed":
        return {k: v.float() for k, v in out.items()}
    return out


# ---------------------------------------------------------------------------
# work: bytes and operations of one pass
def work(case):
    """Bytes: the state (and the table's used share) read and written once per stage.  Operations per
    ordered neighbour pair (the kernel of an unordered pair evaluated once: 15 for r, W and dW; 9 or 10
    for the five kernel sums; 2 dim (dim + dim^2 + ...) for the gradients) and per particle (two table
    evaluations and solves, about 1000; the equations of motion, 500 in 2+1D and 1500 in 3+1D)."""
    if case["kind"] == "serve":
        lo, hi, m = math.log(case["smallest"]), math.log(case["largest"]), case["events"]
        n = sum(math.exp(lo + (hi - lo) * (k + 0.5) / m) for k in range(m))
        w = work({"kind": "bsq2", "n": n, "steps": case["steps"]})
        return {"bytes": w["bytes"] + n * 8 * 20, "flops": w["flops"]}
    kind, n = case["kind"], case["n"]
    d = 3 if kind in ("blob3", "bsq3", "stress3") else 2
    pairs = {"gubser": 72, "bsq2": 285, "diff2": 285, "observe2": 285, "blob3": 280, "bsq3": 600, "stress3": 600}[kind]
    nv = 9 if d == 2 else 13
    stages = 1 if kind == "observe2" else 2 * case["steps"]
    dens, grad = 20.5, 0.0 if kind == "observe2" else (18.0 if d == 2 else 39.0)
    per = 1000.0 + (0.0 if kind == "observe2" else 500.0 if d == 2 else 1500.0)
    if kind == "gubser":
        per = 300.0
    if kind == "diff2":
        grad, per, nv = grad + 24.0, per + 800.0, nv + 6
    return {"bytes": 8.0 * n * stages * 2 * (nv + 7), "flops": stages * n * (pairs * (dens + grad) + per)}


# ---------------------------------------------------------------------------
# the same step in 64 bits, from the equations: kernel sums over explicit pair lists, generic
# four-tensors, the rates' dependence on the acceleration taken by evaluating them at unit vectors
F64 = torch.float64


def _pairs(x, h):
    """Chunks (a, b, r vector, r) of all pairs closer than 2h, the pair of a particle with itself among them."""
    dim, n = x.shape
    c = torch.floor((x - x.min(1, keepdim=True).values) / (2 * h)).long()
    m = c.max(1).values + 3
    mul = torch.tensor([1, int(m[0]), int(m[0] * m[1])][:dim], device=x.device)
    key = ((c + 1) * mul[:, None]).sum(0)
    key, order = torch.sort(key)
    xs = x[:, order]
    for part in torch.arange(n, device=x.device).split(max(1, 40_000_000 // (3 ** dim * (600 if dim == 3 else 300)))):
        for o in range(3 ** dim):
            off = sum(((o // 3 ** k) % 3 - 1) * int(mul[k]) for k in range(dim))
            lo = torch.searchsorted(key, key[part] + off)
            cnt = torch.searchsorted(key, key[part] + off, right=True) - lo
            a = torch.repeat_interleave(part, cnt)
            if a.numel() == 0:
                continue
            start = torch.cumsum(cnt, 0) - cnt
            b = torch.arange(a.numel(), device=x.device) - torch.repeat_interleave(start - lo, cnt)
            r = xs[:, a] - xs[:, b]
            r2 = (r * r).sum(0)
            keep = r2 < (2 * h) * (2 * h)
            a, b, r, r2 = a[keep], b[keep], r[:, keep], r2[keep]
            yield order[a], order[b], r, r2.sqrt()


def _kernel(q, h, dim):
    s = 10.0 / (7.0 * math.pi * h * h) if dim == 2 else 1.0 / (math.pi * h ** 3)
    w = torch.where(q < 1, 1 - 1.5 * q * q + 0.75 * q ** 3, 0.25 * (2 - q) ** 3)
    dw = torch.where(q < 1, -3 * q + 2.25 * q * q, -0.75 * (2 - q) ** 2)
    return s * w, s / h * dw


class _Eos:
    """The closed form, and the quadrilinear table over it."""

    def __init__(self, e, shape):
        self.e, self.t = e, None
        if e.a1 != 0.0:
            k = I.HBARC
            T = torch.linspace(0.05, 0.8, shape[0], dtype=F64, device="cuda") / k
            m = torch.linspace(-0.45, 0.45, shape[1], dtype=F64, device="cuda") / k
            g = torch.meshgrid(T, m, m, m, indexing="ij")
            v = self.closed(g[0].reshape(-1), torch.stack([a.reshape(-1) for a in g[1:]]))
            self.t = torch.cat([v[1], v[0][None]])  # s, n_B, n_S, n_Q, p
            self.shape, self.lo = (shape[0],) + (shape[1],) * 3, torch.stack([T[0], m[0], m[0], m[0]])
            self.hi, self.d = torch.stack([T[-1], m[-1], m[-1], m[-1]]), torch.stack([T[1] - T[0]] + [m[1] - m[0]] * 3)
            self.d = (self.hi - self.lo) / (torch.tensor(self.shape, device="cuda") - 1)

    def closed(self, T, mu):
        """p, (s, n), and the second derivatives [4][4]."""
        e, k = self.e, I.HBARC
        chi = torch.tensor(e.chi, dtype=F64, device=T.device)[:, None]
        th = torch.tanh((T * k - e.Tc_GeV) / e.w_GeV)
        c = k / e.w_GeV
        f, f1, f2 = e.a0 + 0.5 * e.a1 * (1 + th), 0.5 * e.a1 * (1 - th * th) * c, -e.a1 * (1 - th * th) * th * c * c
        q = (chi * mu * mu).sum(0)
        p = T ** 4 * f + 0.5 * T * T * q
        s = 4 * T ** 3 * f + T ** 4 * f1 + T * q
        H = torch.zeros((4, 4) + T.shape, dtype=F64, device=T.device)
        H[0, 0] = 12 * T * T * f + 8 * T ** 3 * f1 + T ** 4 * f2 + q
        for j in range(3):
            H[0, 1 + j] = H[1 + j, 0] = 2 * e.chi[j] * T * mu[j]
            H[1 + j, 1 + j] = e.chi[j] * T * T
        return p, torch.cat([s[None], chi * T * T * mu]), H

    def table(self, x):
        """(s, n, p) of the interpolant and the derivatives of (s, n), [4][4]."""
        r = (x - self.lo[:, None]) / self.d[:, None]
        top = torch.tensor(self.shape, device=x.device)[:, None] - 2
        i = torch.minimum(r.floor().long().clamp(min=0), top)
        t = r - i
        val, der = 0.0, [0.0] * 4
        for c in range(16):
            bit = [(c >> k) & 1 for k in range(4)]
            node = 0
            for k in range(4):
                node = node * self.shape[k] + i[k] + bit[k]
            w = [t[k] if bit[k] else 1 - t[k] for k in range(4)]
            f = self.t[:, node]
            val = val + w[0] * w[1] * w[2] * w[3] * f
            for k in range(4):
                o = [w[j] for j in range(4) if j != k]
                der[k] = der[k] + (1.0 if bit[k] else -1.0) * o[0] * o[1] * o[2] * f[:4]
        return val, torch.stack([der[k] / self.d[k] for k in range(4)], 1)

    def inside(self, x):
        return ((x >= self.lo[:, None]) & (x <= self.hi[:, None])).all(0)

    def newton(self, x, y, tol=1e-13):
        """Damped Newton on the interpolant: the points, and whether they converged."""
        x, s = x.clone(), y[0]
        left, ok = torch.arange(x.shape[1], device=x.device), torch.zeros_like(s, dtype=torch.bool)
        v, J = self.table(x)
        for it in range(30):
            res = ((v[:4] - y[:, left]) / s[left]).abs().max(0).values
            ok[left] = res <= 1e-12
            go = (res > tol) & torch.isfinite(res)
            left, v, J, res = left[go], v[:, go], J[:, :, go], res[go]
            if left.numel() == 0:
                break
            d = torch.linalg.solve(J.permute(2, 0, 1), (y[:, left] - v[:4]).T[..., None])[..., 0].T
            lam, open_ = torch.ones_like(res), torch.ones_like(res, dtype=torch.bool)
            xn, x0 = x[:, left].clone(), x[:, left].clone()
            for _ in range(9):
                tr = torch.minimum(torch.maximum(x0 + lam * d, self.lo[:, None]), self.hi[:, None])
                vt, Jt = self.table(tr)
                good = open_ & (((vt[:4] - y[:, left]) / s[left]).abs().max(0).values < res)
                xn, v, J = torch.where(good, tr, xn), torch.where(good, vt, v), torch.where(good, Jt, J)
                open_ = open_ & ~good
                if not bool(open_.any()):
                    break
                lam = lam * 0.5
            x[:, left] = xn
            keep = ~open_
            left, v, J = left[keep], v[:, keep], J[:, :, keep]
        return x, ok

    def invert(self, y, guess, cap):
        """(s, n) -> T, mu, p, e, (p_s, p_n), d(s, n)/d(T, mu), and the next warm start."""
        e, (s, n) = self.e, (y[0], y[1:])
        chi = torch.tensor([c if c > 0 else 1.0 for c in e.chi], dtype=F64, device=s.device)[:, None]
        c = (n * n / chi).sum(0)
        hi = (s / (4 * e.a0)) ** (1.0 / 3.0)
        lo = hi.clone()

        def g(T):
            return self.closed(T, n / (chi * T * T) if e.chi[0] > 0 else torch.zeros_like(n))[1][0] - s

        last = g(lo)
        none = ~(s > 0)  # no solution: g rises again on the way down, or never changes sign
        for _ in range(400):  # down to a point below the root
            up = (last > 0) & ~none
            if not bool(up.any()):
                break
            lo = torch.where(up, 0.8 * lo, lo)
            now = g(lo)
            none, last = none | (up & (now > last)), torch.where(up, now, last)
        none = none | (last > 0)
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            up = g(mid) > 0
            lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
            if bool((hi - lo <= 3e-16 * hi).all()):
                break
        T = 0.5 * (lo + hi)
        x = torch.cat([T[None], n / (chi * T * T) if e.chi[0] > 0 else torch.zeros_like(n)])
        used = torch.zeros_like(s, dtype=torch.bool)
        if self.t is not None:
            warm = (guess[0] > 0) & self.inside(guess)
            for start, take in ((guess, warm), (x.clone(), ~warm & ~none), (x.clone(), warm & ~none)):
                take = (take & ~used & self.inside(start)).nonzero()[:, 0]
                if take.numel():
                    r, ok = self.newton(start[:, take], y[:, take])
                    x[:, take[ok]], used[take[ok]] = r[:, ok], True
        none = none & ~used
        x[0, none], x[1:, none] = 1.0, 0.0
        p, _, H = self.closed(x[0], x[1:])
        if bool(used.any()):
            v, J = self.table(x[:, used])
            p[used], H[:, :, used] = v[4], J
        act = torch.tensor([True] + [bool(ch > 0) for ch in e.chi], device=s.device) if self.t is None else torch.ones(4, dtype=torch.bool, device=s.device)
        A, z = H.clone(), y.clone()
        for k in range(4):
            if not act[k]:
                A[k], A[:, k], A[k, k], z[k] = 0.0, 0.0, 1.0, 0.0
        Ai = torch.linalg.inv(A.permute(2, 0, 1))
        z = (Ai.transpose(1, 2) @ z.T[..., None])[..., 0].T
        en = (x * y).sum(0) - p
        cs2 = (y * z).sum(0) / (en + p)
        z = torch.where(cs2 > cap, z * (cap / cs2), z)
        wg = torch.where(used, x, torch.cat([-x[:1], torch.zeros_like(x[1:])]))
        p, en, x, z, wg = (torch.where(none, torch.zeros_like(v), v) for v in (p, en, x, z, wg))
        return x, p, en, z, Ai, wg, none


class _Step:
    def __init__(self, e, shape):
        self.e, self.eos, self.dim = e, _Eos(e.eos, shape), e.dim
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", F64)  # noqa: E731
        self.npi = 3 if e.dim == 2 else 5
        df = e.diffusion
        self.diff = df is not None
        rows = [t(e.x), t(e.u), t(e.S)[None], t(e.Bv)[None], t(e.Pv)] + ([torch.zeros((6, e.n), dtype=F64, device="cuda")] if self.diff else [])
        self.y, self.N = torch.cat(rows), t(e.Nq)
        self.tau, self.guess = e.tau0, torch.zeros((4, e.n), dtype=F64, device="cuda")
        if self.diff:
            self.kap, self.tj = torch.tensor(df.kappaT2, dtype=F64, device="cuda"), torch.tensor(df.tauJT, dtype=F64, device="cuda")

    def split(self, y):
        d = self.dim
        return y[:d], y[d:2 * d], y[2 * d], y[2 * d + 1], y[2 * d + 2:2 * d + 2 + self.npi], y[2 * d + 2 + self.npi:]

    def observe(self, y, N, tau):
        """Densities and equation of state at the state y."""
        e, d = self.e, self.dim
        x, u, S, B, P, J = self.split(y)
        n = x.shape[1]
        g = torch.tensor([1.0, -1.0, -1.0, -tau * tau if e.milne else -1.0], dtype=F64, device=x.device)
        U = torch.zeros((4, n), dtype=F64, device=x.device)
        U[1:1 + d] = u
        U[0] = (1 - (g[1:, None] * U[1:] ** 2).sum(0)).sqrt()
        q = torch.cat([torch.ones_like(S)[None], S[None], N])
        sums, nnb = torch.zeros_like(q), torch.zeros(n, dtype=F64, device=x.device)
        for a, b, r, rr in _pairs(x, e.h):
            w = _kernel(rr / e.h, e.h, d)[0]
            for k in range(5):
                sums[k].index_add_(0, a, w * q[k, b])
            nnb.index_add_(0, a, torch.ones_like(w))
        sg = tau if e.milne else 1.0
        star, sig = sums[0], sums[0] / (U[0] * sg)
        dens = sums[1:] / (U[0] * sg)
        if self.diff:
            Jc = sig * J.reshape(3, 2, n)
            J0 = (U[1] * Jc[:, 0] + U[2] * Jc[:, 1]) / U[0]
            dens[1:] = (sums[2:] / sg - J0) / U[0]
        x4, p, en, z, Hi, wg, none = self.eos.invert(dens, self.guess, e.transport.cs2_cap)
        self.guess = wg
        return {"g": g, "U": U, "star": star, "sig": sig, "y4": dens, "x4": x4, "p": p, "e": en, "z": z, "Hi": Hi, "sg": sg, "nnb": nnb, "none": none}

    def full(self, o, st):
        """The 4 x 4 tensor of the stored shear components (any units): traceless and transverse."""
        g, U = o["g"], o["U"]
        pi = torch.zeros((4, 4) + st.shape[1:], dtype=F64, device=st.device)
        at = {(1, 1): 0, (1, 2): 1, (2, 2): 2} if self.dim == 2 else {(1, 1): 0, (1, 2): 1, (1, 3): 2, (2, 2): 3, (2, 3): 4}
        for (i, j), k in at.items():
            pi[i, j] = pi[j, i] = st[k]
        ul = g[:, None] * U
        f = lambda i, j: ul[i] * ul[j] / ul[0] ** 2 + (g[i] if i == j else 0.0)  # noqa: E731
        known = sum(f(i, j) * pi[i, j] for i in (1, 2, 3) for j in (1, 2, 3) if (i, j) != (3, 3))
        pi[3, 3] = -known / f(3, 3)
        for i in (1, 2, 3):
            pi[0, i] = pi[i, 0] = -(ul[1:] * pi[1:, i]).sum(0) / ul[0]
        pi[0, 0] = -(ul[1:] * pi[1:, 0]).sum(0) / ul[0]
        return pi

    def rates(self, y, N, tau):
        e, d, tr = self.e, self.dim, self.e.transport
        o = self.observe(y, N, tau)
        x, u, S, B, P, J = self.split(y)
        g, U, sig, star, sg = o["g"], o["U"], o["sig"], o["star"], o["sg"]
        n, v = x.shape[1], U / U[0]
        if not tr.viscous:
            B, P = torch.zeros_like(B), torch.zeros_like(P)
        Pi, pi = sig * B, self.full(o, sig * P)
        gi = 1 / g
        dlt = torch.diag(gi)
        X = torch.stack([torch.stack([(-(o["p"] + Pi) * gi[j] if i == j else 0.0) + pi[j, i] - v[j] * pi[0, i]
                                      for i in range(1, d + 1)]) for j in range(1, d + 1)]) / star ** 2
        ub = U[1:1 + d] / star
        G, H = torch.zeros((d, n), dtype=F64, device=x.device), torch.zeros((d, n), dtype=F64, device=x.device)
        du = torch.zeros((d, d, n), dtype=F64, device=x.device)  # [k][j] = d_k u^j
        if self.diff:
            Jc = sig * J.reshape(3, 2, n)
            J0 = (U[1] * Jc[:, 0] + U[2] * Jc[:, 1]) / U[0]
            flux = (Jc - v[None, 1:3] * J0[:, None]) / star ** 2
            al = o["x4"][1:] / o["x4"][0]
            dal, div = torch.zeros((3, 2, n), dtype=F64, device=x.device), torch.zeros((3, n), dtype=F64, device=x.device)
        for a, b, r, rr in _pairs(x, e.h):
            far = rr > 0
            a, b, r, rr = a[far], b[far], r[:, far], rr[far]
            dW = _kernel(rr / e.h, e.h, d)[1] * r / rr
            for k in range(d):
                G[k].index_add_(0, a, dW[k])
                H[k].index_add_(0, a, sum(X[j, k, b] * dW[j] for j in range(d)))
                for j in range(d):
                    du[k, j].index_add_(0, a, ub[j, b] * dW[k])
            if self.diff:
                for q in range(3):
                    div[q].index_add_(0, a, ((flux[q][:, a] + flux[q][:, b]) * dW).sum(0))
                    for k in range(2):
                        dal[q, k].index_add_(0, a, (al[q, b] - al[q, a]) * dW[k])
        if self.diff:
            dal = dal / star
        F = -sg * (H + torch.einsum("jin,jn->in", X, G))
        dku = torch.zeros((4, 4, n), dtype=F64, device=x.device)  # d_k u^nu, k = 1..3
        dku[1:1 + d, 1:1 + d] = du
        dku[1:, 0] = -(g[None, 1:, None] * U[None, 1:] * dku[1:, 1:]).sum(1) / U[0]
        Gam = torch.zeros((4, 4, 4), dtype=F64, device=x.device)
        if e.milne:
            Gam[0, 3, 3], Gam[3, 0, 3], Gam[3, 3, 0] = tau, 1 / tau, 1 / tau
        dg3 = -2 * tau if e.milne else 0.0
        (T, mu), (s, nq), z = (o["x4"][0], o["x4"][1:]), (o["y4"][0], o["y4"][1:]), o["z"]
        w, ep = o["e"] + o["p"] + Pi, o["e"] + o["p"]
        Isrc = torch.zeros((4, n), dtype=F64, device=x.device)
        if e.jets is not None:
            for t in e.jets.tracks:
                if tau >= t[6]:
                    c2 = sum((x[k] - t[k] - t[3 + k] * (tau - t[6])) ** 2 for k in range(d))
                    dep = t[7] / ((2 * math.pi) ** 1.5 * e.jets.sigma ** 3) * torch.exp(-c2 / (2 * e.jets.sigma ** 2))
                    Isrc = Isrc + dep * torch.tensor([1.0, t[3], t[4], t[5]], dtype=F64, device=x.device)[:, None]
        eta = tr.eta_over_s * s
        zeta = tr.zeta_peak * torch.exp(-(T * I.HBARC - tr.zeta_T_GeV) ** 2 / (2 * tr.zeta_w_GeV ** 2)) * s
        u0 = U[0]

        def at(acc, Dal):
            """Rates for the acceleration du^i/dx^0 = acc and D alpha = Dal; the equations' residuals."""
            a4 = torch.zeros((4, n), dtype=F64, device=x.device)
            a4[1:1 + d] = acc
            a4[0] = -((g[1:, None] * U[1:] * a4[1:]).sum(0) + 0.5 * dg3 * U[3] ** 2) / u0
            d0u = a4 - (v[1:, None] * dku[1:]).sum(0)
            nab = torch.cat([d0u[None], dku[1:]]) + torch.einsum("cab,bn->acn", Gam, U)
            th = nab[0, 0] + nab[1, 1] + nab[2, 2] + nab[3, 3]
            Du = (U[:, None] * nab).sum(0)
            up = gi[:, None, None] * nab - U[:, None] * Du[None]  # nabla^<mu> u^nu
            Delta = dlt[:, :, None] - U[:, None] * U[None]
            sh = 0.5 * (up + up.transpose(0, 1)) - Delta * th / 3
            dsig = -sig * th / u0
            low = g[:, None] * Du
            pisig = (pi * g[:, None, None] * g[None, :, None] * sh).sum((0, 1))
            dS = (-Pi * th + pisig + (g[:, None] * U * Isrc).sum(0)) / (u0 * sig * T)
            dB, dP = torch.zeros_like(S), torch.zeros_like(pi)
            if tr.viscous:
                tpi = tr.tau_pi_coef * eta / ep
                dB = -(zeta * th + Pi) / (tr.tau_Pi_ratio * tpi * u0 * sig)
                chris = torch.einsum("mn,iml,ljn->ijn", U, Gam, pi)
                coup = U[:, None] * (pi * low[None]).sum(1)[None]
                rhs = (2 * eta * sh - pi) / tpi - 4.0 / 3.0 * pi * th
                dpi = (rhs - chris - chris.transpose(0, 1) - coup - coup.transpose(0, 1)) / u0
                dP = dpi / sig - pi / sig ** 2 * dsig
            dN = torch.zeros((3, n), dtype=F64, device=x.device)
            dJ = None
            if self.diff:
                Jh = J.reshape(3, 2, n)
                jDu = J0 * low[0] + Jc[:, 0] * low[1] + Jc[:, 1] * low[2]
                nabal = -dal - U[None, 1:3] * Dal[:, None]
                src = torch.einsum("qr,rin->qin", self.kap, nabal) * T * T
                DJ = (src - Jc) * T / self.tj[:, None, None] - U[None, 1:3] * jDu[:, None]
                dJ = DJ / (u0 * sig) - Jc / sig ** 2 * dsig
                uJ = (U[None, 1:3] * Jh).sum(1)
                dZ = ((a4[None, 1:3] * Jh + U[None, 1:3] * dJ).sum(1)) / u0 ** 2 - 2 * uJ / u0 ** 3 * a4[0]
                dN = -sg * div - dZ
                dS = dS - (mu * dN).sum(0) / T
            ds = sig * dS + s / sig * dsig
            dn = nq / sig * dsig + sig * dN
            dw = (T + z[0]) * ds + ((mu + z[1:]) * dn).sum(0) + sig * dB + B * dsig
            Ph = pi / sig
            res = []
            for i in range(1, d + 1):
                t1, t2 = 0.0, 0.0
                for j in (1, 2, 3):
                    t1 = t1 + (dg3 if j == 3 else 0.0) * U[j] * Ph[j, i] + g[j] * (a4[j] * Ph[j, i] + U[j] * dP[j, i])
                    t2 = t2 + g[j] * U[j] * Ph[j, i]
                # pi^{0i} / (sigma u^0) = -t2 / u0^2
                dPi0 = -t1 / u0 ** 2 + 2 * t2 / u0 ** 3 * a4[0]
                mom = (U[i] * dw + w * a4[i]) / sig - w * U[i] / sig ** 2 * dsig + dPi0
                T4 = w * U[:, None] * U[None] - (o["p"] + Pi) * dlt[:, :, None] + pi
                src = torch.einsum("ab,abn->n", Gam[i], T4)
                res.append(mom - F[i - 1] + sg * src / star - sg * Isrc[i] / star)
            if self.diff:
                # d alpha / d(s, n) from the inverse Jacobian of (s, n)(T, mu)
                Hi = o["Hi"].permute(1, 2, 0)
                da = (Hi[1:] - mu[:, None] / T * Hi[0][None]) / T
                res += list(Dal - u0 * (da[:, 0] * ds + (da[:, 1:] * dn[None]).sum(1)))
            keep = [(1, 1), (1, 2), (2, 2)] if d == 2 else [(1, 1), (1, 2), (1, 3), (2, 2), (2, 3)]
            f = torch.cat([v[1:1 + d], a4[1:1 + d], dS[None], dB[None], torch.stack([dP[i, j] for i, j in keep])] +
                          ([dJ.reshape(6, n)] if self.diff else []))
            return torch.stack(res), f, dN, (-sg * div if self.diff else None)

        m = d + (3 if self.diff else 0)
        zero = torch.zeros((m, n), dtype=F64, device=x.device)
        r0 = at(zero[:d], zero[d:])[0]
        M = []
        for k in range(m):
            one = zero.clone()
            one[k] = 1.0
            M.append(at(one[:d], one[d:])[0] - r0)
        M = torch.stack(M).permute(2, 1, 0)
        M = torch.where(o["none"][:, None, None], torch.eye(m, dtype=F64, device=x.device), M)
        r0 = torch.where(o["none"], torch.zeros_like(r0), r0)
        sol = torch.linalg.solve(M, -r0.T[..., None])[..., 0].T
        for _ in range(2):  # the affine map's rounding: once more from the solution
            r = torch.where(o["none"], torch.zeros_like(r0), at(sol[:d], sol[d:])[0])
            sol = sol + torch.linalg.solve(M, -r.T[..., None])[..., 0].T
        _, f, dN, dlab = at(sol[:d], sol[d:])
        # no solution, or colder than the stop temperature: ballistic motion alone
        rest = o["none"] | (T * I.HBARC < tr.T_stop_GeV) if tr.T_stop_GeV > 0 else o["none"]
        f[:d, rest], f[d:, rest] = v[1:1 + d, rest], 0.0
        if dlab is not None:
            dlab[:, rest] = 0.0
        return f, dlab

    def step(self):
        dt, y0, N0 = self.e.dtau, self.y, self.N
        f, dN = self.rates(y0, N0, self.tau)
        y1, N1 = y0 + dt * f, N0 if dN is None else N0 + dt * dN
        f, dN = self.rates(y1, N1, self.tau + dt)
        self.y, self.N = 0.5 * (y0 + y1 + dt * f), N0 if dN is None else 0.5 * (N0 + N1 + dt * dN)
        self.tau += dt


def _fields(k, names):
    x, u, S, B, P, J = k.split(k.y)
    got = {"X": x, "U": u, "S": S[None], "NQ": k.N, "BV": B[None], "PV": P, "GUESS": k.guess}
    if "JV" in names:
        got["JV"] = J
    if any(n not in got for n in names):
        warm = k.guess
        o = k.observe(k.y, k.N, k.tau)
        k.guess = warm
        got |= {"SIGMA_STAR": o["star"][None], "S_DENS": o["y4"][:1], "N_DENS": o["y4"][1:], "T": o["x4"][:1], "MU": o["x4"][1:],
                "P": o["p"][None], "E": o["e"][None], "STATUS": None, "NNB": None}
    return {n: got[n] for n in names}


def _table_as_given(k, shape):
    """The table's nodes as the program hands them over (the same doubles)."""
    if k.eos.t is not None:
        t = _table(shape)
        a = [np.ascontiguousarray(v).reshape(-1) for v in (t.s, t.nB, t.nS, t.nQ, t.p)]
        k.eos.t = torch.stack([torch.from_numpy(v).cuda() for v in a])
        k.eos.lo = torch.tensor([t.T0, *t.mu0], dtype=F64, device="cuda")
        k.eos.d = torch.tensor([t.dT, *t.dmu], dtype=F64, device="cuda")
        k.eos.hi = k.eos.lo + k.eos.d * (torch.tensor(k.eos.shape, device="cuda") - 1)
    return k


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        if case["largest"] * case["events"] * case["steps"] > 8_000_000:
            return None  # minutes of pair lists
        state = prepare(case, seed)
        got = []
        for e in state["events"]:
            k = _table_as_given(_Step(e, TABLE), TABLE)
            for _ in range(case["steps"]):
                k.step()
            got.append({n: None if v is None else (v if v.shape[0] > 1 else v[0]) for n, v in _fields(k, SERVED).items()})
        state["server"].free()
        return got
    if case["n"] * (3 if kind in ("bsq3", "stress3") else 1) * case["steps"] > 4_000_000:
        return None  # minutes of pair lists
    e = _event(case, seed)
    k = _table_as_given(_Step(e, _shape(case)), _shape(case))
    for _ in range(0 if kind == "observe2" else case["steps"]):
        k.step()
    if kind == "gubser":
        return {n: v if v.shape[0] > 1 else v[0] for n, v in _fields(k, ("X", "U", "S", "T", "E")).items()}
    return _fields(k, DERIVED if kind == "observe2" else STATE + (("JV",) if kind == "diff2" else ()))
