"""The work that users of this framework have it do, as cases that can be timed and compared.

A case names a lattice (form, boundary, Lx x Ly), a precision and what is done with it:

  step     one qs_trotter_step on the state in hand: the smallest call, a user's own loop
  evolve   |+>^n through a ramp of Trotter steps (qs_evolve), optionally several coupling
           points at once (batch)
  path     a toric-code ground state carried along a parameter path with the energy read
           every few steps (protocol.run_path): the hysteresis, curvature and Trotter-error
           studies
  measure  the observables of a state: norm, energy, loops, fields, Gauss law, density of
           states, fidelity
  grad     final energy of a Fourier schedule and its gradient by autograd (adjoint sweep)
  scan     a phase diagram: many independent coupling points through one schedule, both
           lattices of the scan in one launch (points12 > 0) or one lattice in batches

Observables and gradients of a complex64 state are handed back in single precision, the
precision of the state that they are read from; those of a complex128 state in double.
"""
import math

import numpy as np
import torch

from paper_2108_13410_gb300 import (Simulator, QS_GAUSS, QS_NORM, QS_OPT_GRAPH, QS_OPT_RENORM_EVERY, QS_PLAQUETTE,
                                    QS_THOOFT, QS_WILSON, QS_X)
from paper_2108_13410_gb300.autograd import schedule_value
from paper_2108_13410_gb300.protocol import blue, run_path
from paper_2108_13410_gb300.qsim import qs_scan_mixed

DEVICE = "cuda:0"


def _case(kind, form, Lx, Ly, dtype, boundary="periodic", steps=1, order=2, dt=0.02, batch=1, every=0, points=0,
          points12=0, name=None):
    c = dict(kind=kind, form=form, Lx=Lx, Ly=Ly, boundary=boundary, dtype=dtype, steps=steps, order=order, dt=dt,
             batch=batch, every=every, points=points, points12=points12)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a user's own loop over single steps on the 3x3 torus of the paper's studies (18 qubits)
        _case("step", "ug", 3, 3, "c64", name="step_ug3x3_c64"),
        # the hysteresis and curvature studies: 18 qubits, the energy sampled along the path
        _case("path", "ug", 3, 3, "c64", steps=500, every=125, name="path_ug3x3_c64"),
        # the Trotter-error study of the same lattice, which needs complex128
        _case("path", "ug", 3, 3, "c128", steps=200, every=50, name="path_ug3x3_c128"),
        # the 2x2 torus (12 qubits) compared with exact diagonalisation: T = 10, 100 first-order steps
        _case("evolve", "gh", 2, 2, "c128", steps=100, order=1, dt=0.1, name="evolve_gh2x2_c128"),
        # the headline workload: 27 qubits, a window of the 1000-step ramp
        _case("evolve", "gh", 3, 3, "c64", steps=20, name="evolve_gh3x3_c64"),
        # the same lattice in the paper's precision
        _case("evolve", "gh", 3, 3, "c128", steps=5, name="evolve_gh3x3_c128"),
        # the largest lattice: 4x4 torus, 32 link qubits, 32 GiB
        _case("evolve", "ug", 4, 4, "c64", steps=3, name="evolve_ug4x4_c64"),
        # what is read from a finished 27-qubit run
        _case("measure", "gh", 3, 3, "c64", name="measure_gh3x3_c64"),
        # the same for a 24-qubit run in complex128 (4x3 torus, twelve star operators)
        _case("measure", "ug", 4, 3, "c128", name="measure_ug4x3_c128"),
        # schedule optimisation: many iterations on a lattice of middle size (18 qubits)
        _case("grad", "gh", 3, 2, "c64", steps=100, name="grad_gh3x2_c64"),
        # the adjoint workload's lattice (27 qubits), a shorter schedule
        _case("grad", "gh", 3, 3, "c64", steps=20, name="grad_gh3x3_c64"),
        # a phase diagram of both lattices (12 and 17 qubits) in one launch
        _case("scan", "ug", 3, 2, "c64", boundary="open", steps=100, dt=0.05, batch=304, points=304, points12=304,
              name="scan_12_17_c64"),
    ]


# lattices by form, boundary: sizes that the state of one GPU and the term tables allow
def _lattices(form, max_n, min_n=8):
    found = []
    for boundary in ("periodic", "open"):
        lo = 2 if boundary == "periodic" else 1
        for Lx in range(lo, 9):
            for Ly in range(lo, Lx + 1):
                n, zA, zB, xA, xB, _ = _terms(form, boundary, Lx, Ly)
                if min_n <= n <= max_n and max(len(zA), len(zB), len(xB)) <= 32:
                    found.append((n, boundary, Lx, Ly))
    return sorted(found)


def _pick(rng, found):
    """A lattice, its qubit count (the logarithm of the work) spread evenly over the range."""
    want = rng.choice(sorted({n for n, *_ in found}))
    return rng.choice([f for f in found if f[0] == want])


def draw(rng):
    kind = rng.choice(("step", "evolve", "evolve", "path", "measure", "measure", "grad", "scan"))
    dtype = rng.choice(("c64", "c64", "c128"))
    wide = dtype == "c128"
    form = rng.choice(("gh", "ug"))
    order = rng.choice((1, 2, 2, 2))
    dt = rng.choice((0.01, 0.02, 0.04))
    J = 30 - 2 * wide
    if kind == "path":
        n, b, Lx, Ly = _pick(rng, _lattices("ug", 24 - wide))
        steps = _log(rng, 20, max(20, min(1000, 1 << (32 - n - 2 * wide))))
        return _case("path", "ug", Lx, Ly, dtype, b, steps, order, dt, every=max(1, steps // rng.choice((1, 2, 4))))
    if kind == "grad":
        n, b, Lx, Ly = _pick(rng, _lattices("gh", 24 if wide else 27, 12))
        steps = _log(rng, 3, max(3, min(200, 1 << max(0, 31 - n - 4 * wide))))
        return _case("grad", "gh", Lx, Ly, dtype, b, steps, order, dt)
    if kind == "scan":
        if rng.random() < 0.5:     # both lattices in one launch, a few to some hundred points of each
            p = _log(rng, 16, 400)
            return _case("scan", "ug", 3, 2, "c64", "open", _log(rng, 10, 100), order, 0.05, batch=304,
                         points=p, points12=_log(rng, 1, 400))
        n, b, Lx, Ly = _pick(rng, _lattices(form, 18))
        batch = _log(rng, 1, 32)
        return _case("scan", form, Lx, Ly, dtype, b, _log(rng, 4, 50), order, dt, batch=batch,
                     points=batch * rng.randint(1, 2) - rng.randint(0, batch - 1) // 2)
    n, b, Lx, Ly = _pick(rng, _lattices(form, J))
    if kind == "measure":
        return _case("measure", form, Lx, Ly, dtype, b)
    if kind == "step":
        return _case("step", form, Lx, Ly, dtype, b, 1, order, dt)
    batch = _log(rng, 1, 16) if n <= 20 and rng.random() < 0.4 else 1
    left = 33 - n - 2 * wide - (batch - 1).bit_length()
    return _case("evolve", form, Lx, Ly, dtype, b, _log(rng, 2, max(2, min(400, 1 << max(0, left)))), order, dt, batch)


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# --- inputs ---------------------------------------------------------------------------
def _couplings(case, rng, count):
    if case["kind"] == "scan":
        return [(float(rng.uniform(0.0, 1.5)), float(rng.uniform(0.0, 1.5))) for _ in range(count)]
    J = 0.5 if case["form"] == "ug" else 1.0       # the paper's studies use J = h = 1/2
    return [(float(rng.uniform(0.1, 1.3)), float(rng.uniform(0.1, 1.3)), J, J) for _ in range(count)]


def _ramp(steps, rng):
    """A window of a linear ramp s = t / T, sampled at step midpoints."""
    s0, ds = float(rng.uniform(0.0, 0.4)), float(rng.uniform(0.3, 0.6)) / steps
    return s0 + (np.arange(steps) + 0.5) * ds


def _inputs(case, seed):
    """What both the framework and the 64-bit reference start from, in plain values."""
    rng = np.random.default_rng([seed, 2108])
    kind, steps = case["kind"], case["steps"]
    d = {}
    if kind == "path":
        # a piece of the blue path P -> P', starting at a random place of it
        p = float(rng.uniform(0.12, 0.5))
        whole = blue(p, p / 50000)
        k = int(rng.integers(0, len(whole) - steps))
        d["path"], d["which"] = whole[k:k + steps], int(rng.integers(0, 2))
    elif kind == "grad":
        d["a"] = rng.normal(0.0, 0.01, 16)
        d["cpl"] = _couplings(case, rng, 1)
    elif kind == "scan":
        d["s"] = (np.arange(steps) + 0.5) / steps
        d["points"], d["points12"] = _couplings(case, rng, case["points"]), _couplings(case, rng, case["points12"])
    else:
        d["s"] = _ramp(steps, rng)
        d["cpl"] = _couplings(case, rng, case["batch"])
        d["state_seed"] = int(rng.integers(1 << 31))
        d["s_energy"], d["site"] = float(rng.uniform(0.2, 0.9)), float(rng.uniform())
    return d


def _state(n, seed, dtype, batch=1):
    """A normalised state as a run leaves it: a product of single-qubit states leaning
    towards |+> and |0>, with phases, and a correlated remainder (random amplitudes)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    real = torch.float32 if dtype == "c64" else torch.float64
    rng = np.random.default_rng(seed)
    out = torch.empty((batch, 1 << n), dtype=torch.complex64 if dtype == "c64" else torch.complex128, device=DEVICE)
    for b in range(batch):
        v = out[b]
        torch.randn((1 << n, 2), generator=g, dtype=real, device=DEVICE, out=torch.view_as_real(v))
        v.mul_(0.3 * 2.0 ** (-(n + 1) / 2))
        p = torch.ones(1, dtype=torch.complex128, device=DEVICE)
        for q in range(n):
            th, ph = rng.uniform(0.2, 0.75), rng.uniform(-0.4, 0.4)
            p = torch.cat((p * math.cos(th), p * (math.sin(th) * complex(math.cos(ph), math.sin(ph)))))
            if q == 23 and n > 24:          # the rest of a large state by blocks
                break
        if p.numel() == v.numel():
            v.add_(p.to(v.dtype))
        else:
            rows = v.view(-1, p.numel())
            for r in range(rows.shape[0]):
                rows[r].add_(p.to(v.dtype), alpha=math.sqrt(1.0 / rows.shape[0]))
        v.div_(float(torch.linalg.vector_norm(torch.view_as_real(v).reshape(-1), dtype=torch.float64)))
    return out


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case, d = case, _inputs(case, seed)
    st.__dict__.update(d)
    kind, wide = case["kind"], case["dtype"] == "c128"
    st.sim = Simulator(case["Lx"], case["Ly"], form=case["form"], dtype=case["dtype"], boundary=case["boundary"],
                       batch=case["batch"], device=DEVICE, aux=kind == "grad")
    if kind == "path" and not wide:
        st.sim.set_option(QS_OPT_RENORM_EVERY, 100)      # as the studies do in complex64
    if kind in ("step", "measure"):
        st.sim.state.copy_(_state(st.sim.n, d["state_seed"], case["dtype"], case["batch"]))
    if kind == "measure":
        st.other = _state(st.sim.n, d["state_seed"] + 1, case["dtype"], case["batch"])
    if kind == "grad":
        st.a = torch.tensor(d["a"], dtype=torch.float64 if wide else torch.float32, requires_grad=True)
    if kind == "scan" and case["points12"]:
        st.sim12 = Simulator(2, 2, form="gh", dtype="c64", device=DEVICE)
        st.sim.set_option(QS_OPT_GRAPH, 1)
    torch.cuda.synchronize()
    return st


def _real(case, x):
    """A number or array in the precision of the state that it was read from."""
    return np.asarray(x, dtype=np.float64 if case["dtype"] == "c128" else np.float32)


# --- one pass -------------------------------------------------------------------------
def run(st):
    case, sim = st.case, st.sim
    kind, dt, order = case["kind"], case["dt"], case["order"]
    if kind == "step":
        sim.trotter_step(st.cpl, float(st.s[0]), dt, order)
        return sim.state
    if kind == "evolve":
        sim.init_plus()
        sim.evolve(st.cpl, st.s, dt, order)
        return sim.state
    if kind == "path":
        sim.init_toric(st.which)
        seen = run_path(sim, st.path, dt, order, measure_every=case["every"])
        return {"energy": _real(case, [e for _, e in seen]), "state": sim.state}
    if kind == "measure":
        site = int(st.site * 1000)
        out = {"norm": sim.expect(QS_NORM), "energy": sim.energy(st.cpl), "energy_s": sim.energy(st.cpl, st.s_energy),
               "plaquette": sim.expect(QS_PLAQUETTE, -1), "x": sim.expect(QS_X, site % sim.n), "dos": sim.dos(),
               "fidelity": sim.fidelity(st.other)}
        if case["boundary"] == "periodic":
            out["wilson"] = sim.expect(QS_WILSON, site % 2)
            out["thooft"] = sim.expect(QS_THOOFT, site % 2)
        if case["form"] == "gh":
            out["gauss"] = sim.expect(QS_GAUSS, site % (case["Lx"] * case["Ly"]))
        return {k: _real(case, v) for k, v in out.items()}
    if kind == "grad":
        st.a.grad = None
        v = schedule_value(st.a, sim, st.cpl, dt * case["steps"], case["steps"], order)
        v.backward()
        return {"value": v.detach(), "grad": st.a.grad}
    if case["points12"]:
        o12, o17 = qs_scan_mixed(st.sim12.h, st.points12, sim.h, st.points, st.s, dt, order)
        return {"points12": _real(case, o12), "points": _real(case, o17)}
    return {"points": _real(case, sim.scan(st.points, st.s, dt, order))}


# --- the work that a pass cannot do without -------------------------------------------
def work(case):
    n, zA, zB, xA, xB, _ = _terms(case["form"], case["boundary"], case["Lx"], case["Ly"])
    state = (16 if case["dtype"] == "c128" else 8) * 2 ** n * case["batch"]
    amps = 2 ** n * case["batch"]
    step = 4 * (len(xA) + len(xB)) + 6          # flops per amplitude of one Trotter step
    kind, steps = case["kind"], case["steps"]
    if kind == "step":
        return {"bytes": 2 * state, "flops": amps * step}
    if kind == "evolve":
        return {"bytes": state, "flops": amps * step * steps}
    if kind == "path":
        return {"bytes": state, "flops": amps * step * steps}
    if kind == "measure":
        return {"bytes": 2 * state, "flops": amps * 4 * (len(xA) + len(xB) + 8)}
    if kind == "grad":
        return {"bytes": state, "flops": amps * steps * (3 * step + 4 * (len(xA) + 2))}
    one = case["points"] * 2 ** n * steps * step
    return {"bytes": 64 * (case["points"] + case["points12"]),
            "flops": one + case["points12"] * 4096 * steps * (4 * 12 + 6)}


# --- the same in 64 bits, in plain torch ----------------------------------------------
def _terms(form, boundary, Lx, Ly):
    """(n, plaquettes, bonds or sigma^z, links, vertex X or stars, {loops}) as qubit masks."""
    per = boundary == "periodic"
    vx, vy = (Lx, Ly) if per else (Lx + 1, Ly + 1)
    H, U, q = {}, {}, 0
    for y in range(vy):
        for x in range(vx):
            if per or x + 1 < vx:
                H[x, y] = q
                q += 1
    for y in range(vy):
        for x in range(vx):
            if per or y + 1 < vy:
                U[x, y] = q
                q += 1
    links = q

    def bit(table, x, y):
        k = table.get((x % vx, y % vy) if per else (x, y))
        return 0 if k is None else 1 << k

    verts = [(x, y) for y in range(vy) for x in range(vx)]
    plaq = [bit(H, x, y) | bit(H, x, y + 1) | bit(U, x, y) | bit(U, x + 1, y) for y in range(Ly) for x in range(Lx)]
    stars = [bit(H, x, y) | bit(H, x - 1, y) | bit(U, x, y) | bit(U, x, y - 1) for x, y in verts]
    site = lambda x, y: 1 << (links + (y % vy) * vx + x % vx)  # noqa: E731
    gh = form == "gh"
    ends = {k: site(x, y) | site(x + 1, y) for (x, y), k in H.items()}
    ends.update({k: site(x, y) | site(x, y + 1) for (x, y), k in U.items()})
    second = [(1 << k) | (ends[k] if gh else 0) for k in range(links)]
    n = links + (len(verts) if gh else 0)
    loops = {"stars": stars}
    if per:
        loops["wilson"] = [sum(bit(H, x, 0) for x in range(vx)), sum(bit(U, 0, y) for y in range(vy))]
        loops["thooft"] = [sum(bit(H, 0, y) for y in range(vy)), sum(bit(U, x, 0) for x in range(vx))]
    vertex = [1 << k for k in range(links, n)] if gh else stars
    return n, plaq, second, [1 << k for k in range(links)], vertex, loops


def _flip(psi, mask):
    """X_mask |psi>: amplitude i <- amplitude i ^ mask; psi has shape (batch, 2^n)."""
    shape, dims, left = [psi.shape[0]], [], psi.shape[1].bit_length() - 1
    for k in sorted((k for k in range(left) if mask >> k & 1), reverse=True):
        if left - k - 1:
            shape.append(1 << (left - k - 1))
        dims.append(len(shape))
        shape.append(2)
        left = k
    shape.append(1 << left)
    return torch.flip(psi.view(shape), dims).reshape(psi.shape)


class _Exact:
    def __init__(self, case, form=None, boundary=None, Lx=None, Ly=None):
        self.n, zA, zB, self.xA, self.xB, self.loops = _terms(form or case["form"], boundary or case["boundary"],
                                                               Lx or case["Lx"], Ly or case["Ly"])
        self.nA, self.nB = len(zA), len(zB)
        self.SA, self.SB = self._signs(zA), self._signs(zB)

    def _index(self):
        return torch.arange(1 << self.n, device=DEVICE, dtype=torch.int64)

    def _sign(self, mask):
        i = self._index() & mask
        for k in (32, 16, 8, 4, 2, 1):
            i ^= i >> k
        return 1.0 - 2.0 * (i & 1).to(torch.float32)

    def _signs(self, masks):
        s = torch.zeros(1 << self.n, device=DEVICE, dtype=torch.float32)
        for m in masks:
            s += self._sign(m)
        return s

    # coupling records (g, lambda[, J, h]) as columns
    @staticmethod
    def columns(cpl):
        c = np.array([tuple(x) + (1.0, 1.0)[len(x) - 2:] for x in cpl], dtype=np.float64)
        return tuple(torch.tensor(c[:, k], device=DEVICE)[:, None] for k in range(4))

    def x_layer(self, psi, ta, tb):
        for masks, t in ((self.xA, ta), (self.xB, tb)):
            c, s = torch.cos(t).to(psi.dtype), 1j * torch.sin(t)
            for m in masks:
                f = _flip(psi, m)
                f *= s
                psi = psi.mul_(c).add_(f)
        return psi

    def z_layer(self, psi, za, zb):
        for b in range(psi.shape[0]):
            ph = self.SA.double().mul_(float(za[b])).add_(self.SB.double() * float(zb[b]))
            psi[b].mul_(torch.complex(torch.cos(ph), torch.sin(ph)))
        return psi

    def groups(self, records, dt, order):
        """(X angles, Z angles or None) of each factor group; records: per step (g, l, J, h, s)."""
        out, half = [], None
        for g, lam, J, h, s in records:
            xa, xb = (1 - s) + s * g, (1 - s) + s * J
            z = (s * h * dt, s * lam * dt)
            if order == 1:
                out.append((xa * dt, xb * dt, z))
            else:
                a, b = 0.5 * dt * xa, 0.5 * dt * xb
                out.append((a + half[0], b + half[1], z) if half else (a, b, z))
                half = (a, b)
        if half:
            out.append((half[0], half[1], None))
        return out

    def evolve(self, psi, records, dt, order):
        for a, b, z in self.groups(records, dt, order):
            psi = self.x_layer(psi, a, b)
            if z:
                psi = self.z_layer(psi, *z)
        return psi

    def plus(self, batch):
        return torch.full((batch, 1 << self.n), 2.0 ** (-self.n / 2), dtype=torch.complex128, device=DEVICE)

    def mean(self, psi, mask):
        f = _flip(psi, mask)
        return (torch.view_as_real(psi) * torch.view_as_real(f)).sum((1, 2))

    def parts(self, psi):
        """(norm, <sum Z_A>, <sum Z_B>, <sum X_A>, <sum X_B>) per state."""
        p = torch.view_as_real(psi).square().sum(2)
        za, zb = [torch.stack([(row * s).sum() for row in p]) for s in (self.SA, self.SB)]
        return p.sum(1), za, zb, sum(self.mean(psi, m) for m in self.xA), sum(self.mean(psi, m) for m in self.xB)

    def energy(self, psi, cpl, s=1.0):
        g, lam, J, h = (v[:, 0] for v in self.columns(cpl))
        _, za, zb, xa, xb = self.parts(psi)
        return -(s * h * za + s * lam * zb + ((1 - s) + s * g) * xa + ((1 - s) + s * J) * xb)


def _cost(case):
    """Passes over complex128 memory of the 64-bit run, in bytes."""
    n, zA, zB, xA, xB, _ = _terms(case["form"], case["boundary"], case["Lx"], case["Ly"])
    one = 16.0 * 2 ** n * max(case["batch"], case["points"])
    each = 7 * (len(xA) + len(xB)) + 12
    steps = {"measure": 3, "grad": 4 * case["steps"]}.get(case["kind"], case["steps"] + 1)
    return one * each * steps, one


def exact(case, seed):
    cost, one = _cost(case)
    if cost > 5e13 or one > 2e10:       # over about 20 seconds, or a state that leaves no room
        return None
    d, kind, dt, order = _inputs(case, seed), case["kind"], case["dt"], case["order"]
    E = _Exact(case)
    single = case["dtype"] == "c64"
    if kind in ("step", "evolve"):
        g, lam, J, h = E.columns(d["cpl"])
        psi = _state(E.n, d["state_seed"], case["dtype"], case["batch"]).to(torch.complex128) if kind == "step" \
            else E.plus(case["batch"])
        return E.evolve(psi, [(g, lam, J, h, float(s)) for s in d["s"]], dt, order)
    if kind == "path":
        keep = torch.ones(1 << E.n, dtype=torch.bool, device=DEVICE)
        need = _terms("ug", case["boundary"], case["Lx"], case["Ly"])[1]
        for m in need + (E.loops.get("wilson", []) if d["which"] else []):
            keep &= E._sign(m) > 0
        psi = keep.to(torch.complex128)[None] / math.sqrt(int(keep.sum()))
        energies, path, every = [], d["path"], case["every"]
        for k in range(0, len(path), every):
            piece = path[k:k + every]
            psi = E.evolve(psi, [(*E.columns([c]), 1.0) for c in piece], dt, order)
            energies.append(float(E.energy(psi, [piece[-1]])[0]))
        if single:                       # the framework rescales to unit norm along the way
            psi = psi / torch.linalg.vector_norm(torch.view_as_real(psi))
        return {"energy": np.array(energies), "state": psi}
    if kind == "measure":
        psi = _state(E.n, d["state_seed"], case["dtype"], case["batch"]).to(torch.complex128)
        site = int(d["site"] * 1000)
        norm, za, _, _, _ = E.parts(psi)
        p = torch.view_as_real(psi).square().sum(2)
        links = sum(E._signs([m]) for m in E.xA)
        k = ((len(E.xA) - links) / 2).round().to(torch.int64)
        dos = torch.stack([torch.zeros(len(E.xA) + 1, dtype=torch.float64, device=DEVICE).index_add_(0, k, row)
                           for row in p])
        out = {"norm": norm, "energy": E.energy(psi, d["cpl"]), "energy_s": E.energy(psi, d["cpl"], d["s_energy"]),
               "plaquette": za / E.nA, "x": E.mean(psi, 1 << (site % E.n)), "dos": dos}
        if case["boundary"] == "periodic":
            out["wilson"] = (p * E._sign(E.loops["wilson"][site % 2])).sum(1)
            out["thooft"] = E.mean(psi, E.loops["thooft"][site % 2])
        if case["form"] == "gh":
            v = site % (case["Lx"] * case["Ly"])
            out["gauss"] = E.mean(psi, E.loops["stars"][v] | E.xB[v])
        other = _state(E.n, d["state_seed"] + 1, case["dtype"], case["batch"]).to(torch.complex128)
        out["fidelity"] = (other.conj() * psi).sum(1).abs().square()
        return {k: v.cpu().numpy() for k, v in out.items()}
    if kind == "grad":
        return _exact_grad(case, d, E)
    s = [float(x) for x in d["s"]]

    def points(E, pts):
        out = []
        room = max(1, int(4e9 / (16 * 2 ** E.n)))
        for k in range(0, len(pts), room):
            part = pts[k:k + room]
            g, lam, J, h = E.columns(part)
            psi = E.evolve(E.plus(len(part)), [(g, lam, J, h, x) for x in s], dt, order)
            norm, za, zb, xa, xb = E.parts(psi)
            e = -(h[:, 0] * za + lam[:, 0] * zb + g[:, 0] * xa + J[:, 0] * xb)
            zero = torch.zeros_like(norm)
            w = [(torch.view_as_real(psi).square().sum(2) * E._sign(m)).sum(1) for m in E.loops.get("wilson", [])]
            gh = len(E.xB) and E.n > len(E.xA)
            out.append(torch.stack([e, za / max(1, E.nA), *(w or [zero, zero]), norm, xa / len(E.xA),
                                    xb / len(E.xB) if gh else zero, zero], 1))
        return torch.cat(out).cpu().numpy()

    if case["points12"]:
        return {"points12": points(_Exact(case, "gh", "periodic", 2, 2), d["points12"]), "points": points(E, d["points"])}
    return {"points": points(E, d["points"])}


def _exact_grad(case, d, E):
    """Energy after the schedule s(t) = t/T + sum_m a_m sin(m pi t / T) and its gradient in a."""
    N, dt, order = case["steps"], case["dt"], case["order"]
    a = d["a"].astype(np.float32 if case["dtype"] == "c64" else np.float64).astype(np.float64)
    T = dt * N
    t = (np.arange(1, N + 1) - 0.5) * (T / N)
    jac = np.sin(np.outer(np.arange(1, 17), t) * math.pi / T)
    s = t / T + a @ jac
    g, lam, J, h = (float(v[0, 0]) for v in E.columns(d["cpl"]))
    col = lambda x: torch.tensor([[x]], dtype=torch.float64, device=DEVICE)  # noqa: E731
    rec = [(g, lam, J, h, x) for x in s]
    groups = E.groups(rec, dt, order)
    psi = E.plus(1)
    for xa, xb, z in groups:
        psi = E.x_layer(psi, col(xa), col(xb))
        if z:
            psi = E.z_layer(psi, [z[0]], [z[1]])
    lamb = -(h * E.SA + lam * E.SB).double() * psi
    for masks, c in ((E.xA, g), (E.xB, J)):
        for m in masks:
            lamb -= c * _flip(psi, m)
    value = float((psi.conj() * lamb).sum().real)
    im = lambda f: float((lamb.conj() * f).sum().imag)  # noqa: E731
    ds = np.zeros(N)
    for j in reversed(range(len(groups))):
        xa, xb, z = groups[j]
        if z:
            ds[j] += -2.0 * dt * (h * im(E.SA * psi) + lam * im(E.SB * psi))
            psi, lamb = E.z_layer(psi, [-z[0]], [-z[1]]), E.z_layer(lamb, [-z[0]], [-z[1]])
        gx = -2.0 * ((g - 1.0) * sum(im(_flip(psi, m)) for m in E.xA) + (J - 1.0) * sum(im(_flip(psi, m)) for m in E.xB))
        if order == 1:
            ds[j] += gx * dt
        else:
            if j < N:
                ds[j] += gx * 0.5 * dt
            if j:
                ds[j - 1] += gx * 0.5 * dt
        psi, lamb = E.x_layer(psi, col(-xa), col(-xb)), E.x_layer(lamb, col(-xa), col(-xb))
    return {"value": value, "grad": jac @ ds}
