"""The work that programs have this library do, as cases that can be timed and compared.

A case is one periodic water-like box (atoms O, H, H per molecule at 0.0334 molecules per
cubic Angstrom, charge widths 0.70 / 0.45 A, seeded noise on every parameter) and one of the
calls below.  ``listed`` holds the sizes of this library's own configurations (648, 3,000,
24,000 and 300,000 atoms, a served mix of 100 to 20,000) and ``draw`` the range between them:
ragged molecule counts, orthorhombic boxes, cutoffs, spline orders and both precisions.

kinds
    apply     System.apply: potential, field, force and energies of given charges
    grad      coulomb_energy, forward and backward: an energy inside a trained model
    evaluate  new positions: neighbour build, then one shadow evaluation (a served request)
    md        a segment of a trajectory: state in, ``steps`` shadow steps, state out
    solve     qeq_solve: charges of the regular (Born-Oppenheimer) form by GMRES
    batch     the served form of md: several systems of mixed size, stepped together

FP32-mixed results carry single precision (the mode's error is about 1e-6), and programs that
choose it keep and pass on float32: trajectory frames, model inputs, gradients of float32
leaves.  ``run`` returns them so; FP64 results stay float64.
"""

import math

import numpy as np
import torch

import paper_2503_21176_gb300 as qg

K_E = 14.3996454784
ALPHA, SKIN = 0.34, 1.0
MASS_UNIT = 103.6427
RANK, K_D, DT = 2, 5, 0.5
KINDS = ("apply", "grad", "evaluate", "md", "solve", "batch")


def _case(kind, n_mol, precision, r_cut=8.0, order=4, spacing=1.01, steps=0, aspect=1.0, short=False,
          count=1, min_mol=0, name=None):
    c = {"kind": kind, "n_mol": n_mol, "precision": precision, "r_cut": r_cut, "order": order,
         "spacing": spacing, "steps": steps, "aspect": aspect, "short": short, "count": count,
         "min_mol": min_mol}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration (216 molecules, r_c 9, mesh 32^3): launches and latency
        _case("apply", 216, "fp64", r_cut=9.0, spacing=0.6, name="apply 648 fp64"),
        # a ragged orthorhombic box at a tighter accuracy (order 6), the default precision
        _case("apply", 7411, "fp64", order=6, aspect=1.25, spacing=1.2, name="apply 22k fp64 order 6"),
        # the headline box: Coulomb applies in both precisions
        _case("apply", 100_000, "fp32_mixed", name="apply 300k fp32"),
        _case("apply", 100_000, "fp64", name="apply 300k fp64"),
        # training through the energy: the 24,000-atom differentiation box
        _case("grad", 8000, "fp32_mixed", name="grad 24k fp32"),
        # a served request on new positions, of ordinary size
        _case("evaluate", 1000, "fp32_mixed", name="evaluate 3k fp32"),
        # the same on the headline box: the neighbour build counts most
        _case("evaluate", 100_000, "fp32_mixed", name="evaluate 300k fp32"),
        # a trajectory of the smallest configuration, with the built-in short-range model
        _case("md", 216, "fp64", r_cut=9.0, spacing=0.6, steps=20, short=True, name="md 648 fp64"),
        # the headline shadow-MD steps (list rebuilds among them), and their FP64 form
        _case("md", 100_000, "fp32_mixed", steps=16, name="md 300k fp32"),
        _case("md", 100_000, "fp64", steps=3, name="md 300k fp64"),
        # start charges of a trajectory: the iterative solve
        _case("solve", 6667, "fp64", name="solve 20k fp64"),
        # eight requests of the served mix, 100 to 20,000 atoms, stepped as one batch
        _case("batch", 6667, "fp32_mixed", steps=10, count=8, min_mol=34, name="batch 8 fp32"),
    ]


def draw(rng):
    kind = rng.choice(KINDS)
    precision = rng.choice(("fp64", "fp32_mixed"))
    # largest boxes: what each kind is run at (FP64 trajectories and solves are kept smaller)
    top = {"apply": 100_000, "grad": 60_000, "evaluate": 100_000, "solve": 12_000, "batch": 6667}
    top["md"] = 40_000 if precision == "fp64" else 80_000
    n_mol = int(round(math.exp(rng.uniform(math.log(40), math.log(top[kind])))))
    steps, count, min_mol = 0, 1, 0
    if kind == "md":
        steps = rng.randint(2, 6)
    if kind == "batch":
        steps, count, min_mol = rng.randint(2, 6), rng.randint(2, 8), 34
        n_mol = max(n_mol, 80)
    return _case(kind, n_mol, precision, r_cut=round(rng.uniform(7.0, 9.0), 2), order=rng.choice((4, 4, 5, 6)),
                 spacing=round(rng.uniform(0.7, 1.2), 2), steps=steps, aspect=round(rng.uniform(0.85, 1.3), 3),
                 short=kind in ("md", "batch") and rng.random() < 0.3, count=count, min_mol=min_mol)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _box(case, n_mol):
    """Edges of the box: (aspect, 1, 1 / aspect) times the cubic edge."""
    L = (n_mol / 0.0334) ** (1.0 / 3.0)
    return L * case["aspect"], L, L / case["aspect"]


def _mesh(case, box):
    """The smallest even 2-3-5-7-smooth sizes with at most the case's spacing."""
    def smooth(k):
        for f in (2, 3, 5, 7):
            while k % f == 0:
                k //= f
        return k == 1

    mesh = []
    for L in box:
        k = max(int(math.ceil(L / case["spacing"])), case["order"], 4)
        while k % 2 or not smooth(k):
            k += 1
        mesh.append(k)
    return tuple(mesh)


def _water(case, n_mol, seed):
    """Seeded arrays of one box (numpy float64), positions not wrapped."""
    rng = np.random.default_rng([int(seed), n_mol])
    box = np.array(_box(case, n_mol))
    a = (box.prod() / n_mol) ** (1.0 / 3.0)
    sides = [int(math.ceil(L / a - 1e-9)) for L in box]
    cell = box / sides
    sites = rng.permutation(sides[0] * sides[1] * sides[2])[:n_mol]
    grid = np.stack(np.unravel_index(sites, sides), axis=1)
    oxy = (grid + 0.5 + rng.uniform(-0.1, 0.1, (n_mol, 3))) * cell
    half = math.radians(104.52) / 2
    quat = rng.standard_normal((n_mol, 4))
    w, x, y, z = (quat / np.linalg.norm(quat, axis=1, keepdims=True)).T
    ax = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], axis=1)
    az = np.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], axis=1)
    R = np.empty((n_mol, 3, 3))
    R[:, 0] = oxy
    R[:, 1] = oxy + 0.9572 * (math.sin(half) * ax + math.cos(half) * az)
    R[:, 2] = oxy + 0.9572 * (-math.sin(half) * ax + math.cos(half) * az)
    R = R.reshape(-1, 3)
    n = 3 * n_mol
    is_o = np.arange(n) % 3 == 0
    mass = np.where(is_o, 15.999, 1.008)
    V = rng.standard_normal((n, 3)) * np.sqrt(0.025852 / (mass[:, None] * MASS_UNIT))
    V -= (mass[:, None] * V).sum(0) / mass.sum()
    q = 0.4 * rng.standard_normal(n)
    n0 = np.where(is_o, -0.16, 0.08) + 0.01 * rng.standard_normal(n)  # near the water charges
    return {"R": R, "V": V, "mass": mass, "q": q - q.mean(), "n0": n0 - n0.mean(),
            "chi": np.where(is_o, 8.5, 4.5) + 0.1 * rng.standard_normal(n),
            "eta": np.where(is_o, 14.0, 12.0) + 0.1 * rng.standard_normal(n),
            "sigma": np.where(is_o, 0.70, 0.45) * (1 + 0.02 * rng.uniform(-1, 1, n)), "box": box}


def _members(case):
    """Molecules of each system of the case (one, or a batch spread over its range)."""
    if case["count"] == 1:
        return [case["n_mol"]]
    lo, hi, k = case["min_mol"], case["n_mol"], case["count"]
    return [int(round(lo * (hi / lo) ** (i / (k - 1)))) for i in range(k)]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _inputs(case, seed):
    """[{name: tensor}] of each system, on the GPU; the box stays on the host."""
    out = []
    for k, n_mol in enumerate(_members(case)):
        w = _water(case, n_mol, seed * 16 + k)
        out.append({name: a if name == "box" else torch.as_tensor(a, dtype=torch.float64, device=_device())
                    for name, a in w.items()})
    return out


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

STATE = ("R", "V", "F", "Kf", "n_hist")


def _system(case, w):
    return qg.System(qg.make_params(
        w["R"].shape[0], w["box"], alpha=ALPHA, r_cut=case["r_cut"], skin=SKIN, mesh=_mesh(case, w["box"]),
        order=case["order"], precision=case["precision"], k_e=K_E, krylov_rank=RANK, dissipation_k=K_D, dt=DT,
        short_range=qg.QEQ_SHORT_WATER if case["short"] else qg.QEQ_SHORT_NONE, mass_unit=MASS_UNIT))


def prepare(case, seed):
    """The system of each box with its list, the inputs, and for trajectories the evaluated state."""
    # steps are captured into graphs on a stream of the program's own
    state = {"case": case, "stream": torch.cuda.Stream()}
    with torch.cuda.stream(state["stream"]):
        state["w"] = _inputs(case, seed)
        state["sys"] = [_system(case, w) for w in state["w"]]
        kind = case["kind"]
        if kind != "evaluate":
            for s, w in zip(state["sys"], state["w"]):
                s.neighbor_build(w["R"])
        if kind in ("evaluate", "md", "batch"):
            state["md"] = [qg.ShadowMD(s, w["chi"], w["eta"], w["sigma"], w["mass"], w["R"], w["V"], w["n0"])
                           for s, w in zip(state["sys"], state["w"])]
        if kind in ("md", "batch"):
            for md in state["md"]:
                md.init()
            state["now"] = [getattr(md, k) for md in state["md"] for k in STATE]
            state["from"] = [t.clone() for t in state["now"]]
            state["batch"] = qg.ShadowBatch() if kind == "batch" else None
        if kind == "grad":
            w = state["w"][0]
            t = torch.float32 if case["precision"] == "fp32_mixed" else torch.float64
            # the leaves a single-precision model has; the list is that of the positions it passes on
            state["leaves"] = [w[k].to(t).requires_grad_() for k in ("q", "R")]
            state["sys"][0].neighbor_build(state["leaves"][1].detach().double())
    torch.cuda.synchronize()
    return state


def _out(case, out):
    if case["precision"] == "fp32_mixed":
        return {k: v.float() for k, v in out.items()}
    return out


def run(state):
    with torch.cuda.stream(state["stream"]):
        return _run(state)


def _run(state):
    case, kind = state["case"], state["case"]["kind"]
    w, sysm = state["w"][0], state["sys"][0]
    if kind == "apply":
        v, E, F, energy = sysm.apply(w["R"], w["q"], w["sigma"])
        return _out(case, {"v": v, "E": E, "F": F, "energy": energy})
    if kind == "grad":
        q, R = state["leaves"]
        e = qg.coulomb_energy(sysm, R.double(), q.double(), w["sigma"])
        gq, gR = torch.autograd.grad(e, (q, R))
        return _out(case, {"energy": e.detach(), "gq": gq, "gR": gR})
    if kind == "solve":
        q = torch.zeros_like(w["chi"])
        info = qg.qeq_solve(sysm.ctx, w["R"], w["chi"], w["eta"], w["sigma"], q, 1e-8)
        return _out(case, {"q": q, "lambda": torch.tensor(info["lambda"], dtype=torch.float64)})
    if kind == "evaluate":
        md = state["md"][0]
        sysm.neighbor_build(md.R)
        md.init()
        return _out(case, {"q": md.q, "F": md.F, "Kf": md.Kf, "energies": md.energies})
    # trajectories: the state comes in, takes its steps, and is the result
    torch._foreach_copy_(state["now"], state["from"])
    if kind == "md":
        state["md"][0].step(case["steps"])
    else:
        for _ in range(case["steps"]):
            state["batch"].step(state["md"])
    out = {}
    for k, md in enumerate(state["md"]):
        out |= {"%s%d" % (name, k): t for name, t in (("R", md.R), ("V", md.V), ("F", md.F), ("q", md.q),
                                                      ("n", md.n_hist[0]), ("energies", md.energies))}
    return _out(case, out)


def work(case):
    """Inputs read and outputs written once; 40 flops per directed pair inside the cutoff, the spline
    weights' spread and gather, and two real transforms per Coulomb operator."""
    bytes_, flops = 0.0, 0.0
    for n_mol in _members(case):
        n = 3 * n_mol
        K = math.prod(_mesh(case, _box(case, n_mol)))
        pairs = n * 4.0 / 3.0 * math.pi * case["r_cut"] ** 3 * 3 * 0.0334
        apply_ = 40.0 * pairs + n * case["order"] ** 3 * 12.0 + 2 * 2.5 * K * math.log2(K)
        kind = case["kind"]
        if kind in ("apply", "grad"):
            b, f = 96.0 * n if kind == "apply" else 72.0 * n, apply_
        elif kind == "solve":
            b, f = 56.0 * n, 15 * apply_
        elif kind == "evaluate":
            # 4.6 candidate distances (8 flops) for each entry inside r_cut + skin
            b = 104.0 * n
            f = (RANK + 1) * apply_ + 8 * 4.6 * pairs * (1 + SKIN / case["r_cut"]) ** 3
        else:
            b, f = (24 + 24 + 24 + 8 + 8 * (K_D + 1)) * 2.0 * n + 40.0 * n, case["steps"] * (RANK + 1) * apply_
        bytes_ += b
        flops += f
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

class _Operator:
    """Phi at fixed positions: pair sum over every image inside the cutoff, smooth PME, self terms."""

    def __init__(self, case, w, R):
        dev = R.device
        self.n, self.rc, self.order = R.shape[0], case["r_cut"], case["order"]
        self.box = torch.as_tensor(w["box"], dtype=torch.float64, device=dev)
        self.sigma = w["sigma"]
        x = R - self.box * torch.floor(R / self.box)
        self.i, self.j, d = self._pairs(x)
        self.d = d if case["short"] else None
        r = d.norm(dim=1)
        gamma = torch.sqrt(self.sigma[self.i] ** 2 + self.sigma[self.j] ** 2)
        two = 2 / math.sqrt(math.pi)
        self.f, df = torch.zeros_like(r), torch.zeros_like(r)
        for a, sign in ((torch.full_like(r, ALPHA), 1.0), (1 / gamma, -1.0)):
            e = torch.special.erfc(a * r) / r
            self.f += sign * e
            df -= sign * (e + two * a * torch.exp(-((a * r) ** 2))) / r
        self.g = d * (df / r)[:, None]
        self._splines(x, _mesh(case, w["box"]))

    def _pairs(self, x):
        L, rc = self.box, self.rc
        if bool((L < 3 * rc).any()):  # every atom against every image
            reach = [int(math.ceil(rc / float(v))) for v in L]
            parts = []
            for s in np.ndindex(*(2 * m + 1 for m in reach)):
                shift = torch.tensor([a - m for a, m in zip(s, reach)], dtype=x.dtype, device=x.device) * L
                for lo in range(0, self.n, 4096):
                    d = x[None] - x[lo:lo + 4096, None] + shift
                    ok = (d * d).sum(-1) < rc * rc
                    if not bool(shift.any()):
                        k = torch.arange(d.shape[0], device=x.device)
                        ok[k, lo + k] = False
                    a, b = ok.nonzero(as_tuple=True)
                    parts.append((a + lo, b, d[a, b]))
            return [torch.cat(p) for p in zip(*parts)]
        nc = [int(float(v) / rc) for v in L]
        ncell = math.prod(nc)
        c3 = [torch.clamp((x[:, k] / L[k] * nc[k]).long(), max=nc[k] - 1) for k in range(3)]
        cell = (c3[0] * nc[1] + c3[1]) * nc[2] + c3[2]
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=ncell)
        first = torch.cumsum(count, 0) - count
        most = int(count.max())
        table = torch.full((ncell, most), -1, dtype=torch.long, device=x.device)
        slot = torch.arange(self.n, device=x.device) - first[cell[order]]
        table[cell[order], slot] = order
        at = torch.arange(ncell, device=x.device)
        a3 = (at // (nc[1] * nc[2]), at // nc[2] % nc[1], at % nc[2])
        step = max(1, 12_000_000 // most ** 2)
        parts = []
        for o in np.ndindex(3, 3, 3):
            u = [a3[k] + o[k] - 1 for k in range(3)]
            s = [torch.div(u[k], nc[k], rounding_mode="floor") for k in range(3)]
            other = ((u[0] - s[0] * nc[0]) * nc[1] + u[1] - s[1] * nc[1]) * nc[2] + u[2] - s[2] * nc[2]
            shift = torch.stack(s, 1).to(x.dtype) * L
            for lo in range(0, ncell, step):
                ia, ib = table[lo:lo + step], table[other[lo:lo + step]]
                d = (x[ib] + shift[lo:lo + step, None])[:, None] - x[ia][:, :, None]
                ok = ((d * d).sum(-1) < rc * rc) & (ia >= 0)[:, :, None] & (ib >= 0)[:, None]
                if o == (1, 1, 1):
                    ok &= ia[:, :, None] != ib[:, None]
                p, a, b = ok.nonzero(as_tuple=True)
                parts.append((ia[p, a], ib[p, b], d[p, a, b]))
        return [torch.cat(p) for p in zip(*parts)]

    def _splines(self, x, K):
        p, dev = self.order, x.device
        self.K = K
        u = x * (torch.tensor(K, dtype=torch.float64, device=dev) / self.box)
        base = torch.floor(u)
        w = u - base
        M = torch.zeros(p, *w.shape, dtype=torch.float64, device=dev)  # M[j] = M_n(w + j)
        M[0], M[1] = w, 1 - w
        zero = torch.zeros_like(w)
        for n in range(3, p + 1):
            old = M.clone()
            if n == p:
                self.dM = torch.stack([(old[j] if j < p - 1 else zero) - (old[j - 1] if j else zero)
                                       for j in range(p)])
            for j in range(n):
                left, right = (old[j] if j < n - 1 else zero), (old[j - 1] if j else zero)
                M[j] = ((w + j) * left + (n - w - j) * right) / (n - 1)
        self.M = M
        at = [[(base[:, k].long() - j) % K[k] for j in range(p)] for k in range(3)]
        self.point = [(a, b, c, (at[0][a] * K[1] + at[1][b]) * K[2] + at[2][c]) for a in range(p)
                      for b in range(p) for c in range(p)]
        ints = [0.0, 1.0] + [0.0] * (p - 2)  # M_n at 0, 1, 2, ...
        for n in range(3, p + 1):
            ints = [(j * (ints[j] if j < n - 1 else 0.0) + (n - j) * (ints[j - 1] if j else 0.0)) / (n - 1)
                    for j in range(n)] + [0.0] * (p - n)
        b2, k2 = [], []
        for k in range(3):
            m = torch.arange(K[k], dtype=torch.float64, device=dev)
            ph = 2 * math.pi / K[k] * torch.remainder(m[:, None] * torch.arange(p - 1, device=dev), K[k])
            Mk = torch.tensor(ints[1:p], dtype=torch.float64, device=dev)
            den = (Mk * torch.cos(ph)).sum(1) ** 2 + (Mk * torch.sin(ph)).sum(1) ** 2
            b2.append(torch.where(den > 1e-10, 1 / den, torch.zeros_like(den)))
            mm = torch.where(m <= K[k] // 2, m, m - K[k])
            k2.append((2 * math.pi * mm / self.box[k]) ** 2)
        h = K[2] // 2 + 1
        kk = k2[0][:, None, None] + k2[1][:, None] + k2[2][:h]
        G = K_E * 4 * math.pi / float(self.box.prod()) * torch.exp(-kk / (4 * ALPHA ** 2)) / kk
        G[0, 0, 0] = 0
        self.G = G * b2[0][:, None, None] * b2[1][:, None] * b2[2][:h]

    def apply(self, q):
        """v, E and the energy parts (total, real space, mesh, self)."""
        n, K = self.n, self.K
        vr = K_E * torch.zeros_like(q).index_add_(0, self.i, self.f * q[self.j])
        E = K_E * torch.zeros(n, 3, dtype=q.dtype, device=q.device).index_add_(0, self.i, self.g * q[self.j][:, None])
        mesh = torch.zeros(math.prod(K), dtype=q.dtype, device=q.device)
        for a, b, c, at in self.point:
            mesh.index_add_(0, at, q * self.M[a][:, 0] * self.M[b][:, 1] * self.M[c][:, 2])
        phi = torch.fft.irfftn(self.G * torch.fft.rfftn(mesh.view(K)), s=K).reshape(-1) * math.prod(K)
        vm, Em = torch.zeros_like(q), torch.zeros_like(E)
        for a, b, c, at in self.point:
            ph = phi[at]
            mx, my, mz = self.M[a][:, 0], self.M[b][:, 1], self.M[c][:, 2]
            vm += ph * mx * my * mz
            Em[:, 0] -= ph * self.dM[a][:, 0] * my * mz
            Em[:, 1] -= ph * mx * self.dM[b][:, 1] * mz
            Em[:, 2] -= ph * mx * my * self.dM[c][:, 2]
        E += Em * (torch.tensor(K, dtype=q.dtype, device=q.device) / self.box)
        vs = K_E * (math.sqrt(2 / math.pi) / self.sigma - 2 * ALPHA / math.sqrt(math.pi)) * q
        v = vr + vm + vs
        return v, E, torch.stack([0.5 * q @ v, 0.5 * q @ vr, 0.5 * mesh @ phi, 0.5 * q @ vs])


def _short(case, w, R, op):
    """Energy of the flexible-water model (SPC/Fw bonds, angle, O-O Lennard-Jones inside the cutoff)."""
    kcal = 0.0433641
    m = R.view(-1, 3, 3)
    a, b = ((d - op.box * torch.round(d / op.box)) for d in (m[:, 1] - m[:, 0], m[:, 2] - m[:, 0]))
    ra, rb = a.norm(dim=1), b.norm(dim=1)
    theta = torch.acos((a * b).sum(1) / (ra * rb))
    e = 0.5 * 1059.162 * kcal * ((ra - 0.9572) ** 2 + (rb - 0.9572) ** 2).sum()
    e = e + 0.5 * 75.90 * kcal * ((theta - math.radians(104.52)) ** 2).sum()
    oo = (op.i % 3 == 0) & (op.j % 3 == 0)
    i, j = op.i[oo], op.j[oo]
    with torch.no_grad():  # the pair's image: the list's displacement less the difference of the positions
        shift = op.box * torch.round((op.d[oo] - (R[j] - R[i])) / op.box)
    d2 = ((R[j] - R[i] + shift) ** 2).sum(1)
    s6 = 3.165492 ** 6 / d2 ** 3
    return e + 0.5 * (4 * 0.1554 * kcal * (s6 * s6 - s6)).sum()


class _Shadow:
    """The shadow evaluation and step of one system."""

    def __init__(self, case, w):
        self.case, self.w = case, w
        self.R, self.V = w["R"].clone(), w["V"].clone()
        self.hist = [w["n0"].clone() for _ in range(K_D + 1)]

    def evaluate(self):
        w, n = self.w, self.hist[0]
        op = _Operator(self.case, w, self.R)
        iu = 1 / w["eta"]
        v, En, _ = op.apply(n)
        lam = -((w["chi"] + v) * iu).sum() / iu.sum()
        q = -(w["chi"] + v + lam) * iu
        f = q - n
        phi, Ef, _ = op.apply(f)
        self.F = q[:, None] * En + n[:, None] * Ef
        e_short = torch.zeros((), dtype=q.dtype, device=q.device)
        if self.case["short"]:
            Rg = self.R.clone().requires_grad_()
            e = _short(self.case, w, Rg, op)
            self.F = self.F - torch.autograd.grad(e, Rg)[0]
            e_short = e.detach()
        W, Rb = [f / f.norm()], []
        pw = phi / f.norm()
        for k in range(RANK):
            mu = -(pw * iu).sum() / iu.sum()
            Rb.append(-(pw + mu) * iu - W[k])
            if k + 1 < RANK:
                x = Rb[k].clone()
                for y in W:
                    x = x - (x @ y) * y
                W.append(x / x.norm())
                pw = op.apply(W[-1])[0]
        B = torch.stack(Rb)
        self.Kf = torch.linalg.solve(B @ B.T, B @ f) @ torch.stack(W)
        self.q = q
        self.energies = torch.stack([torch.zeros_like(lam), q @ w["chi"] + 0.5 * (w["eta"] * q * q).sum() + q @ v
                                     - 0.5 * n @ v + e_short, torch.zeros_like(lam), e_short, lam, q.sum(), f.norm(),
                                     torch.full_like(lam, RANK + 1.0)])
        self._kinetic()

    def _kinetic(self):
        self.energies[0] = 0.5 * MASS_UNIT * (self.w["mass"][:, None] * self.V ** 2).sum()
        self.energies[2] = self.energies[0] + self.energies[1]

    def step(self):
        hk = (DT / (2 * MASS_UNIT) / self.w["mass"])[:, None]
        self.V = self.V + hk * self.F
        self.R = self.R + DT * self.V
        c = (-6, 14, -8, -3, 4, -1)
        n = 2 * self.hist[0] - self.hist[1] - 1.82 * self.Kf
        n = n + 18e-3 * sum(ck * h for ck, h in zip(c, self.hist))
        self.hist = [n] + self.hist[:-1]
        self.evaluate()
        self.V = self.V + hk * self.F
        self._kinetic()


def exact(case, seed):
    kind = case["kind"]
    ws = _inputs(case, seed)
    w = ws[0]
    if kind in ("apply", "grad"):
        q, R = w["q"], w["R"]
        if kind == "grad" and case["precision"] == "fp32_mixed":
            q, R = q.float().double(), R.float().double()
        v, E, energy = _Operator(case, w, R).apply(q)
        F = q[:, None] * E
        return {"v": v, "E": E, "F": F, "energy": energy} if kind == "apply" else \
            {"energy": energy[0], "gq": v, "gR": -F}
    if kind == "solve":  # conjugate gradients on the neutral subspace, eliminating lambda
        op, u, chi = _Operator(case, w, w["R"]), w["eta"], w["chi"]
        A = lambda x: u * x + op.apply(x)[0]  # noqa: E731
        P = lambda x: x - x.mean()  # noqa: E731
        q = torch.zeros_like(chi)
        r = P(-chi)
        p, rr = r, r @ r
        r0 = rr
        for _ in range(300):
            if rr <= 1e-26 * r0:
                break
            Ap = P(A(p))
            a = rr / (p @ Ap)
            q, r = q + a * p, r - a * Ap
            new = r @ r
            p, rr = r + (new / rr) * p, new
        return {"q": q, "lambda": -(chi + A(q)).mean()}
    shadows = [_Shadow(case, x) for x in ws]
    out = {}
    for k, s in enumerate(shadows):
        s.evaluate()
        for _ in range(case["steps"]):
            s.step()
        if kind == "evaluate":
            return {"q": s.q, "F": s.F, "Kf": s.Kf, "energies": s.energies}
        out |= {"%s%d" % (name, k): t for name, t in (("R", s.R), ("V", s.V), ("F", s.F), ("q", s.q),
                                                      ("n", s.hist[0]), ("energies", s.energies))}
    return out
