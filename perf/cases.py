"""Performance cases of the public entry points.

A case is a dict of plain values:

* ``kind``     "apply" (ed_apply_H), "propagate" (ed_propagate), "ground"
               (ed_ground_state), "spectral" (ed_spectral_propagate) or "docc"
               (ed_double_occupation),
* ``lattice``  "ring:L", "chain:L", "ladder:L" (2 x L) or "torus:LxxLy",
* ``n_up``, ``n_dn``, ``U``, ``dtype`` ("c64" or "c128"),
* ``disorder`` width of seeded random on-site energies (0: none),
* apply: ``nvec`` vectors per call, ``field`` magnitude of the static vector
  potential,
* propagate and spectral: ``m``, ``steps`` time steps per call; propagate also
  ``tol`` (> 0: adaptive Krylov dimension), ``scheme`` ("midpoint" or
  "cfet4"), ``energy`` (record E(t) as well).

States are normalised complex normal vectors whose amplitudes fall by a factor
per doubly occupied site, like those of a state of a repulsive lattice.  The
pulse is that of the benchmark, entered near its peak.
"""
import math

import numpy as np
import torch

import synth
from paper_2005_13498_gb300 import ed

DT = 0.02
DOUBLON = 0.45      # amplitude factor per doubly occupied site of the start states
PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 10.0}
T_START = 9.0       # near the peak of the pulse
SPECTRAL_PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0}


def _case(name, kind, lattice, n_up, n_dn, dtype, **more):
    c = {"name": name, "kind": kind, "lattice": lattice, "n_up": n_up, "n_dn": n_dn,
         "dtype": dtype, "U": 8.0, "disorder": 0.0}
    if kind == "apply":
        c.update(nvec=1, field=0.3)
    if kind in ("propagate", "spectral"):
        c.update(m=20, steps=1)
    if kind == "propagate":
        c.update(tol=0.0, scheme="midpoint", energy=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest product: an 8-site ring, where only latency counts
        _case("apply_ring8_c128", "apply", "ring:8", 4, 4, "c128"),
        # a short trajectory with its energy on the smallest workload
        _case("steps_ring8_c128", "propagate", "ring:8", 4, 4, "c128", m=12, steps=20,
              energy=True),
        # trajectories on the 12-site square lattice, in both precisions; in
        # double precision with the fourth-order scheme and energies
        _case("steps_torus12_c64", "propagate", "torus:4x3", 6, 6, "c64", steps=10),
        _case("steps_torus12_c128", "propagate", "torus:4x3", 6, 6, "c128", steps=2,
              scheme="cfet4", energy=True),
        # the 14-site ladder at half filling, the headline workload, in the
        # precision a long run uses and in the one it is checked with
        _case("steps_ladder14_c64", "propagate", "ladder:7", 7, 7, "c64", m=30, steps=2),
        _case("step_ladder14_c128", "propagate", "ladder:7", 7, 7, "c128", m=30),
        # the same ladder with the adaptive Krylov dimension
        _case("adaptive_ladder14_c64", "propagate", "ladder:7", 7, 7, "c64", m=30, steps=4,
              tol=1e-8, energy=True),
        # one product in the one-hole sector: rows of 3003 elements
        _case("apply_ladder14_hole_c64", "apply", "ladder:7", 7, 6, "c64"),
        # the largest sector, 16 sites at half filling: vectors beyond the L2
        _case("apply_torus16_c64", "apply", "torus:4x4", 8, 8, "c64"),
        # Green's functions: 48 c / c+ states and the state itself, one batch
        _case("spectral_torus12_c64", "spectral", "torus:4x3", 6, 6, "c64", steps=2),
        # the ground state a propagation starts from, with site energies
        _case("ground_torus12_c128", "ground", "torus:4x3", 6, 5, "c128", disorder=0.4),
        # the double occupancy of a given state, average and per site
        _case("docc_ladder14_c128", "docc", "ladder:7", 7, 7, "c128"),
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "propagate", "propagate", "propagate",
                       "propagate", "spectral", "ground", "docc"])
    dtype = rng.choice(["c64", "c128"])
    lo, hi = {"apply": (4e3, 1.2e7), "propagate": (4e3, 1.2e7), "spectral": (4e3, 4e5),
              "ground": (4e3, 8e5), "docc": (4e3, 1.2e7)}[kind]
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for _ in range(60):     # the sector whose dimension is nearest to the target
        shape = rng.choice(["ring", "chain", "ladder", "torus"])
        if shape == "torus":
            lat, Ns = rng.choice([("torus:3x3", 9), ("torus:4x3", 12)])
        elif shape == "ladder":
            L = rng.randint(4, 7)
            lat, Ns = "ladder:%d" % L, 2 * L
        else:
            Ns = rng.randint(8, 14)
            lat = "%s:%d" % (shape, Ns)
        nu, nd = rng.randint(2, Ns - 2), rng.randint(2, Ns - 2)
        D = math.comb(Ns, nu) * math.comb(Ns, nd)
        if kind == "ground" and (abs(nu - nd) != 1 or abs(nu + nd - Ns) > 1):
            # near half filling, where a gap separates the ground state; with
            # equal numbers spin-flip partners would share the largest element
            continue
        if lo <= D <= hi:
            off = abs(math.log(D / target))
            if best is None or off < best[0]:
                best = (off, lat, nu, nd, D)
    _, lat, nu, nd, D = best or (0, "ladder:5", 5, 4, 52920)
    c = _case("", kind, lat, nu, nd, dtype, U=round(rng.uniform(2.0, 10.0), 2))
    del c["name"]
    if kind == "ground":
        c.update(dtype="c128", disorder=0.4)
    elif rng.random() < 0.25:
        c["disorder"] = 0.3
    if kind == "apply":
        c.update(nvec=rng.choice([1, 1, 2, 3]), field=rng.choice([0.0, 0.3]))
    if kind in ("propagate", "spectral"):
        c["m"] = rng.randint(8, 30 if kind == "propagate" else 20)
    if kind == "propagate":
        c["steps"] = max(1, min(20, int(3e7 / (D * (4 if dtype == "c128" else 1)))))
        c.update(tol=rng.choice([0.0, 0.0, 1e-7]), scheme=rng.choice(["midpoint", "cfet4"]),
                 energy=rng.choice([False, True]))
    return c


# ------------------------------------------------------------------ inputs
def _lattice(case, seed):
    shape, size = case["lattice"].split(":")
    if shape == "torus":
        lat = synth.torus(*[int(x) for x in size.split("x")])
    else:
        lat = {"ring": synth.ring, "chain": synth.chain, "ladder": synth.ladder}[shape](int(size))
    lat = dict(lat)
    if case["disorder"]:
        r = np.random.default_rng(seed + 77)
        lat["eps"] = case["disorder"] * r.uniform(-1.0, 1.0, lat["Ns"])
    return lat


def _pulse(case):
    p = dict(PULSE if case["kind"] == "propagate" else SPECTRAL_PULSE)
    p["dir"] = (1.0, 1.0, 0.0) if case["lattice"].startswith("torus") else (1.0, 0.0, 0.0)
    return p


def _field(case):
    return [case["field"], 0.5 * case["field"], 0.0]


def _words(Ns, n):
    w = np.arange(1 << Ns, dtype=np.int64)
    bits = np.zeros_like(w)
    for i in range(Ns):
        bits += (w >> i) & 1
    return w[bits == n]


def _doublons(Ns, up, dn, dev):
    """Number of doubly occupied sites of every element, int8 [up, dn]."""
    u = torch.from_numpy(up).to(dev)
    d = torch.from_numpy(dn).to(dev)
    out = torch.zeros((len(up), len(dn)), dtype=torch.int8, device=dev)
    for i in range(Ns):
        out += (((u >> i) & 1)[:, None] * ((d >> i) & 1)[None, :]).to(torch.int8)
    return out


def _states(Ns, up, dn, count, seed, dtype, dev):
    """count seeded normalised states, complex128 or complex64 [count, D]."""
    weight = torch.tensor(DOUBLON, dtype=torch.float64, device=dev) ** torch.arange(
        Ns + 1, dtype=torch.float64, device=dev)
    D = len(up) * len(dn)
    out = torch.empty((count, D), dtype=torch.complex64 if dtype == "c64" else torch.complex128,
                      device=dev)
    nd = _doublons(Ns, up, dn, dev).reshape(-1)
    g = torch.Generator(device=dev).manual_seed(seed)
    for k in range(count):
        x = torch.randn(D, dtype=torch.complex128, device=dev, generator=g)
        for a in range(0, D, 1 << 24):      # in pieces: int64 indices of 2^24 elements
            x[a:a + (1 << 24)] *= weight[nd[a:a + (1 << 24)].long()]
        out[k] = x / torch.linalg.vector_norm(x)
    return out


def prepare(case, seed):
    dev = torch.device("cuda")
    lat = _lattice(case, seed)
    Ns, nu, nd, dtype = lat["Ns"], case["n_up"], case["n_dn"], case["dtype"]
    h = ed.Hubbard(lat, nu, nd, case["U"])
    up, dn = _words(Ns, nu), _words(Ns, nd)
    s = {"case": dict(case), "h": h, "Ns": Ns, "seed": seed,
         "dtype": ed.ED_C64 if dtype == "c64" else ed.ED_C128}
    if case["kind"] == "apply":
        s["v"] = _states(Ns, up, dn, case["nvec"], seed, dtype, dev)
        s["w"] = torch.zeros_like(s["v"])
        ed.ed_set_field(h.ctx, _field(case))
    elif case["kind"] == "propagate":
        s["psi0"] = _states(Ns, up, dn, 1, seed, dtype, dev)[0].contiguous()
        s["psi"] = torch.zeros_like(s["psi0"])
        s["pulse"] = _pulse(case)
        ed.ed_set_krylov_tol(h.ctx, case["tol"])
        ed.ed_set_integrator(h.ctx, case["scheme"])
    elif case["kind"] == "spectral":
        s["psi0"] = _states(Ns, up, dn, 1, seed, "c128", dev)[0].contiguous()
        s["pulse"] = _pulse(case)
    elif case["kind"] == "docc":
        s["psi"] = _states(Ns, up, dn, 1, seed, dtype, dev)[0].contiguous()
    else:
        s["psi"] = torch.zeros(h.D, dtype=torch.complex128, device=dev)
    return s


def _real(x, case):
    """Numbers computed from complex64 vectors are good to single precision."""
    x = np.asarray(x)
    if case["dtype"] == "c128":
        return x
    return x.astype(np.complex64 if x.dtype.kind == "c" else np.float32)


def run(state):
    c, h, dtype = state["case"], state["h"], state["dtype"]
    if c["kind"] == "apply":
        ed.ed_apply_H(h.ctx, state["v"], state["w"], dtype, nvec=c["nvec"])
        return state["w"]
    if c["kind"] == "propagate":
        state["psi"].copy_(state["psi0"])
        o = ed.ed_propagate(h.ctx, state["psi"], dtype, state["pulse"], T_START, DT, c["steps"],
                            c["m"], energy=c["energy"])
        out = {"psi": state["psi"], "docc": _real(o["docc"], c), "norm2": _real(o["norm2"], c),
               "m_eff": o["m_eff"]}
        if c["energy"]:
            out["energy"] = _real(o["energy"], c)
        if c["tol"]:        # with a fixed dimension the estimate is rounding
            out["delta"] = _real(o["delta"], c)
        return out
    if c["kind"] == "spectral":
        less, great = ed.ed_spectral_propagate(h.ctx, state["psi0"], dtype, state["pulse"], DT,
                                               c["steps"], c["m"], state["Ns"])
        return {"less": _real(less, c), "great": _real(great, c)}
    if c["kind"] == "docc":
        d, site = ed.ed_double_occupation(h.ctx, state["psi"], dtype)
        return {"docc": d, "site": site[:state["Ns"]]}
    E, _ = ed.ed_ground_state(h.ctx, state["psi"], tol=1e-12, max_iter=3000, seed=state["seed"] + 1)
    return {"E0": E, "psi": state["psi"]}


# -------------------------------------------------------------------- work
def _hops(lat, n):
    """Mean number of allowed hops into a configuration of one spin."""
    Ns = lat["Ns"]
    pairs = math.comb(Ns - 2, n - 1) if 1 <= n <= Ns - 1 else 0
    return 2.0 * len(lat["p"]) * pairs / math.comb(Ns, n)


def work(case):
    """Bytes: the state(s) in and out.  Operations of a product: the two
    additions of every hop and the multiply-add of the diagonal; of a Lanczos
    step also the two inner products and the two vector updates."""
    lat = _lattice(case, 0)
    Ns, nu, nd = lat["Ns"], case["n_up"], case["n_dn"]
    D = math.comb(Ns, nu) * math.comb(Ns, nd)
    size = 8 if case["dtype"] == "c64" else 16
    hv = D * (2.0 * (_hops(lat, nu) + _hops(lat, nd)) + 4.0)
    if case["kind"] == "apply":
        return {"bytes": 2.0 * D * size * case["nvec"], "flops": hv * case["nvec"]}
    if case["kind"] == "docc":
        return {"bytes": 1.0 * D * size, "flops": 4.0 * D}
    if case["kind"] == "ground":
        return {"bytes": 1.0 * D * size, "flops": 60.0 * (hv + 16.0 * D)}
    steps = case["steps"] * (2 if case.get("scheme") == "cfet4" else 1)
    m = 8 if case.get("tol") else case["m"]
    step = m * (hv + 16.0 * D) + 8.0 * m * D
    if case["kind"] == "spectral":
        return {"bytes": 16.0 * D, "flops": (4 * Ns + 1) * steps * step}
    return {"bytes": 2.0 * D * size, "flops": steps * step}


# ------------------------------------------------------------------- exact
class _Model:
    """The Hamiltonian of one sector in 64 bits, by lists of neighbours."""

    def __init__(self, case, seed, nu, nd, dev):
        lat = _lattice(case, seed)
        self.Ns, self.dev = lat["Ns"], dev
        self.p, self.q = [int(x) for x in lat["p"]], [int(x) for x in lat["q"]]
        self.t, self.d = np.asarray(lat["t"]), np.asarray(lat["d"]).reshape(-1, 3)
        self.words = [_words(self.Ns, nu), _words(self.Ns, nd)]
        self.double = _doublons(self.Ns, self.words[0], self.words[1], dev)
        self.U = case["U"]
        eps = lat.get("eps")
        self.eps = [None if eps is None else torch.from_numpy(
            sum(eps[i] * ((w >> i) & 1) for i in range(self.Ns))).to(dev) for w in self.words]
        self.hops = [self._hop_list(w) for w in self.words]

    def _hop_list(self, words):
        """Per bond and direction: the targets, their sources and the signs."""
        out = []
        for b, (p, q) in enumerate(zip(self.p, self.q)):
            lo, hi = min(p, q), max(p, q)
            between = np.zeros(len(words), dtype=np.int64)
            for i in range(lo + 1, hi):
                between += (words >> i) & 1
            sign = 1.0 - 2.0 * (between & 1)
            for a, c, way in ((p, q, 0), (q, p, 1)):      # an electron from a to c
                t = np.nonzero(((words >> c) & 1 == 1) & ((words >> a) & 1 == 0))[0]
                src = np.searchsorted(words, words[t] ^ (1 << a) ^ (1 << c))
                out.append((b, way, t, src, sign[t]))
        return out

    def tables(self, coef):
        """Padded neighbour lists of both spins for hop coefficients coef[b]
        (the reverse hop has the conjugate)."""
        tabs = []
        for words, hops in zip(self.words, self.hops):
            dim = len(words)
            fill = np.zeros(dim, dtype=np.int64)
            width = max(1, int(np.bincount(np.concatenate([h[2] for h in hops]),
                                           minlength=dim).max()) if hops else 1)
            nbr = np.zeros((width, dim), dtype=np.int64)
            val = np.zeros((width, dim), dtype=np.complex128)
            for b, way, t, src, sign in hops:
                nbr[fill[t], t] = src
                val[fill[t], t] = sign * (coef[b] if way == 0 else np.conj(coef[b]))
                fill[t] += 1
            tabs.append((torch.from_numpy(nbr).to(self.dev), torch.from_numpy(val).to(self.dev)))
        return tabs

    def bond_coef(self, A):
        return -self.t * np.exp(-1j * (self.d @ np.asarray(A, dtype=np.float64)))

    def apply(self, tabs, x):
        """H x for x of shape [up, dn], complex128."""
        w = x * (self.U * self.double)
        if self.eps[0] is not None:
            w += x * self.eps[0][:, None]
            w += x * self.eps[1][None, :]
        for k in range(tabs[0][0].shape[0]):
            w += tabs[0][1][k][:, None] * x[tabs[0][0][k]]
        for k in range(tabs[1][0].shape[0]):
            w += tabs[1][1][k][None, :] * x.index_select(1, tabs[1][0][k])
        return w


def _dot(a, b):
    return torch.sum(a.conj() * b)


def _small_exp(al, be, tau):
    n = len(al)
    T = np.diag(al) + np.diag(be[:n - 1], 1) + np.diag(be[:n - 1], -1)
    lam, Q = np.linalg.eigh(T)
    return Q @ (np.exp(-1j * tau * lam) * Q[0])


def _krylov(model, tabs, x, tau, m, tol):
    """exp(-i tau H) x from m Lanczos vectors, or as many as the adaptive
    exit takes; with the estimate delta and the dimension."""
    b0 = float(torch.linalg.vector_norm(x))
    V, al, be, old, scale = [x / b0], [], [], np.zeros(0), 1.0
    delta = 0.0
    for j in range(1, m + 1):
        w = model.apply(tabs, V[-1])
        if j > 1:
            w -= be[-1] * V[-2]
        al.append(float(_dot(V[-1], w).real))
        if j == m:
            break
        w -= al[-1] * V[-1]
        be.append(float(torch.linalg.vector_norm(w)))
        if tol > 0:
            y = _small_exp(np.array(al), np.array(be), tau)
            ny = float(np.linalg.norm(y))
            delta = float(np.linalg.norm(y - np.append(old, np.zeros(len(y) - len(old))))) / ny
            err = min(1 + ny, delta / (1 - delta) * ny) if delta < 1 else 1 + ny
            scale = max(scale, abs(al[-1]))
            if err < tol or be[-1] < tol * scale:
                break
            scale = max(scale, be[-1])
            old = y
        V.append(w / be[-1])
    y = _small_exp(np.array(al), np.array(be), tau)
    if tol > 0 and len(al) == m:
        delta = float(np.linalg.norm(y - np.append(old, 0))) / float(np.linalg.norm(y))
    out = torch.zeros_like(x)
    for yj, v in zip(y, V):
        out += b0 * complex(yj) * v
    return out, delta, len(al)


def _amplitude(pulse, t):
    s = t - pulse["t0"]
    a = pulse["A0"] * math.exp(-s * s / (2 * pulse["sigma"] ** 2)) * math.sin(pulse["omega"] * s)
    return a * np.asarray(pulse["dir"])


def _substeps(model, pulse, t, scheme):
    """(tables, length) of the exponentials of one time step from t, in the
    order they act."""
    if scheme == "midpoint":
        return [(model.tables(model.bond_coef(_amplitude(pulse, t + DT / 2))), DT)]
    r = math.sqrt(3.0)
    c1 = model.bond_coef(_amplitude(pulse, t + (0.5 - r / 6) * DT))
    c2 = model.bond_coef(_amplitude(pulse, t + (0.5 + r / 6) * DT))
    a1, a2 = (3 - 2 * r) / 12, (3 + 2 * r) / 12
    return [(model.tables(2 * (a2 * c1 + a1 * c2)), DT / 2),
            (model.tables(2 * (a1 * c1 + a2 * c2)), DT / 2)]


def _exact_propagate(case, seed, dev):
    model = _Model(case, seed, case["n_up"], case["n_dn"], dev)
    pulse = _pulse(case)
    up, dn = model.words
    x = _states(model.Ns, up, dn, 1, seed, case["dtype"], dev)[0].to(torch.complex128)
    x = x.reshape(len(up), len(dn))
    out = {"docc": [], "norm2": [], "energy": [], "delta": [], "m_eff": None}

    def observe(t):
        q = x.real ** 2 + x.imag ** 2
        out["norm2"].append(float(q.sum()))
        out["docc"].append(float((q * model.double).sum()) / model.Ns)
        if case["energy"]:
            tabs = model.tables(model.bond_coef(_amplitude(pulse, t)))
            out["energy"].append(float(_dot(x, model.apply(tabs, x)).real) / model.Ns)

    observe(T_START)
    for n in range(case["steps"]):
        deltas = []
        for tabs, tau in _substeps(model, pulse, T_START + n * DT, case["scheme"]):
            x, delta, _ = _krylov(model, tabs, x, tau, case["m"], case["tol"])
            deltas.append(delta)
        out["delta"].append(max(deltas))
        observe(T_START + (n + 1) * DT)
    got = {k: np.array(out[k]) for k in ("docc", "norm2")}
    if case["energy"]:
        got["energy"] = np.array(out["energy"])
    if case["tol"]:
        got["delta"] = np.array(out["delta"])
    return dict(got, psi=x.reshape(-1), m_eff=None)


def _fermion(Ns, words, target, site, create, before):
    """Targets, sources and signs of c or c+ at one site on one spin's words;
    before: electrons of the other spin ordered in front."""
    bit = 1 << site
    t = np.nonzero(((target & bit) != 0) == create)[0]
    x = target[t] ^ bit
    below = np.full(len(t), before)
    for i in range(site):
        below += (x >> i) & 1
    return t, np.searchsorted(words, x), 1.0 - 2.0 * (below & 1)


def _exact_spectral(case, seed, dev):
    base = _Model(case, seed, case["n_up"], case["n_dn"], dev)
    Ns, pulse, nu, nd = base.Ns, _pulse(case), case["n_up"], case["n_dn"]
    up, dn = base.words
    psi0 = _states(Ns, up, dn, 1, seed, "c128", dev)[0].reshape(len(up), len(dn))
    steps = case["steps"]

    def walk(model, x):
        xs = [x]
        for n in range(steps):
            for tabs, tau in cached(model, n):
                x = _krylov(model, tabs, x, tau, case["m"], 0.0)[0]
            xs.append(x)
        return xs

    memo = {}

    def cached(model, n):
        key = (id(model), n)
        if key not in memo:
            memo[key] = _substeps(model, pulse, n * DT, "midpoint")
        return memo[key]

    psis = walk(base, psi0)
    G = [np.zeros((steps + 1, Ns, 2), dtype=np.complex128) for _ in range(2)]
    keep = []
    for op in range(2):
        for spin in range(2):
            k = 1 if op else -1
            tu, td = (nu + k, nd) if spin == 0 else (nu, nd + k)
            if not (0 <= tu <= Ns and 0 <= td <= Ns):
                continue
            model = _Model(case, seed, tu, td, dev)
            keep.append(model)
            for site in range(Ns):
                t, src, sign = _fermion(Ns, base.words[spin], model.words[spin], site, op == 1,
                                        nu if spin == 1 else 0)
                t, src = torch.from_numpy(t).to(dev), torch.from_numpy(src).to(dev)
                sign = torch.from_numpy(sign).to(dev)

                def op_on(x):
                    y = torch.zeros((len(model.words[0]), len(model.words[1])),
                                    dtype=torch.complex128, device=dev)
                    if spin == 0:
                        y[t] = x[src] * sign[:, None]
                    else:
                        y[:, t] = x[:, src] * sign[None, :]
                    return y

                for n, phi in enumerate(walk(model, op_on(psi0))):
                    ov = complex(_dot(op_on(psis[n]), phi))
                    G[op][n, site, spin] = 1j * ov if op == 0 else -1j * ov
    return {"less": G[0], "great": G[1]}


def _exact_ground(case, seed, dev):
    model = _Model(case, seed, case["n_up"], case["n_dn"], dev)
    tabs = model.tables(model.bond_coef([0.0, 0.0, 0.0]))
    shape = (len(model.words[0]), len(model.words[1]))
    g = torch.Generator(device=dev).manual_seed(1)
    x = torch.randn(shape, dtype=torch.complex128, device=dev, generator=g)
    x /= torch.linalg.vector_norm(x)
    E = 0.0
    for _ in range(30):         # restarted Lanczos with full reorthogonalisation
        V, al, be = [x], [], []
        for _ in range(min(120, shape[0] * shape[1])):
            w = model.apply(tabs, V[-1])
            al.append(float(_dot(V[-1], w).real))
            Q = torch.stack(V).reshape(len(V), -1)
            w = w.reshape(-1)
            for _ in range(2):
                w = w - Q.T @ (Q.conj() @ w)
            be.append(float(torch.linalg.vector_norm(w)))
            if be[-1] < 1e-12:
                break
            V.append((w / be[-1]).reshape(shape))
        n = len(al)
        T = np.diag(al) + np.diag(be[:n - 1], 1) + np.diag(be[:n - 1], -1)
        s = np.linalg.eigh(T)[1][:, 0]
        x = sum(float(c) * v for c, v in zip(s, V))
        x /= torch.linalg.vector_norm(x)
        hx = model.apply(tabs, x)
        E = float(_dot(x, hx).real)
        if float(torch.linalg.vector_norm(hx - E * x)) < 2e-13 * max(1.0, abs(E)):
            break
    x = x.reshape(-1)
    top = x[torch.argmax(x.abs())]
    return {"E0": E, "psi": x * (top.conj() / top.abs())}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "propagate":
        return _exact_propagate(case, seed, dev)
    if case["kind"] == "spectral":
        return _exact_spectral(case, seed, dev)
    if case["kind"] == "ground":
        return _exact_ground(case, seed, dev)
    model = _Model(case, seed, case["n_up"], case["n_dn"], dev)
    up, dn = model.words
    x = _states(model.Ns, up, dn, case.get("nvec", 1), seed, case["dtype"], dev)
    if case["kind"] == "docc":
        x = x[0].to(torch.complex128).reshape(len(up), len(dn))
        q = x.real ** 2 + x.imag ** 2
        u, d = torch.from_numpy(up).to(dev), torch.from_numpy(dn).to(dev)
        site = [float(((u >> i) & 1).to(q) @ q @ ((d >> i) & 1).to(q)) for i in range(model.Ns)]
        return {"docc": sum(site) / model.Ns, "site": np.array(site)}
    tabs = model.tables(model.bond_coef(_field(case)))
    w = torch.empty(x.shape, dtype=torch.complex128, device=dev)
    for k in range(x.shape[0]):
        w[k] = model.apply(tabs, x[k].to(torch.complex128).reshape(len(up), len(dn))).reshape(-1)
    return w
