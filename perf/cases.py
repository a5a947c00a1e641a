"""What a user of this framework has it do, as cases that can be timed and checked.

Every case goes through the public entry points (Engine, Mlp).  Five kinds:

  evolve   Engine.run from the initial operator: Trotter steps, double-layer BP and
           the correlator after each, on growing bond dimensions.
  layer    one Trotter layer, BP and the correlator on a saturated state (every bond
           at chi_max), restarted from a device snapshot.
  bp       double-layer BP alone on a saturated state: all converged messages.
  measure  the correlator alone (single-layer BP, Bethe sums, Pauli weights).
  train    one gradient and Adam step of the learned warm start.

BP runs a fixed sweep budget (the tolerance is out of reach), so that a pass is the
same work whatever the last bits of its messages; after a Trotter step it is about what
the usual tolerance of 1e-5 takes, or more.  Results of the FP32-storage modes are handed
over in FP32, the type that they are computed to.  The signs of singular vectors are
free (a degenerate pair's whole rotation is), so a Trotter step hands over what does not
depend on them: the spectra of every bond, the Pauli weights of every site and the
measured scalars.
"""
import math
import random

import numpy as np
import torch

import paper_2606_30985_gb300 as pkg

DECAY = 0.06          # lambda_k ~ exp(-DECAY k): a saturated Schmidt spectrum
WEIGHT = (1.0, 0.5, 0.5, 0.5)
OUT_OF_REACH = 1e-30  # BP tolerance: the sweep budget ends every BP run
EPS_CUT = 1e-11


def listed():
    return [
        # the smallest study: 3x3, FP64, first-order steps from the initial operator
        dict(name="evolve_3x3_chi8_fp64", kind="evolve", Lx=3, Ly=3, chi=8, prec="fp64", order=1, steps=5, sweeps=20, n=1),
        # the 4x4 off-centre study in the default precision
        dict(name="evolve_4x4_chi20_fp32", kind="evolve", Lx=4, Ly=4, chi=20, prec="fp32", order=2, steps=6, sweeps=20, n=1),
        # a scan over fields: instances of mixed sizes batched in one engine
        dict(name="evolve_batch9_fp32", kind="evolve", Lx=4, Ly=4, chi=16, prec="fp32", order=2, steps=4, sweeps=18, n=9),
        # saturated layers: full precision, default precision with an odd chi on a ragged
        # grid, the default precision's larger studies, the tensor-core mode
        dict(name="layer_4x4_chi12_fp64", kind="layer", Lx=4, Ly=4, chi=12, prec="fp64", order=2, sweeps=26),
        dict(name="layer_3x5_chi27_fp32", kind="layer", Lx=3, Ly=5, chi=27, prec="fp32", order=2, sweeps=18),
        dict(name="layer_4x4_chi48_fp32", kind="layer", Lx=4, Ly=4, chi=48, prec="fp32", order=2, sweeps=18),
        dict(name="layer_4x4_chi64_tf32x3", kind="layer", Lx=4, Ly=4, chi=64, prec="tf32x3", order=2, sweeps=18),
        # the benchmark's bond dimension on the smallest grid with an interior site
        dict(name="layer_3x3_chi100_tf32x3", kind="layer", Lx=3, Ly=3, chi=100, prec="tf32x3", order=2, sweeps=18),
        # BP alone, as a trap retry runs it: the benchmark's chi, and the default precision
        dict(name="bp_3x4_chi100_tf32x3", kind="bp", Lx=3, Ly=4, chi=100, prec="tf32x3", sweeps=3),
        dict(name="bp_5x5_chi32_fp32", kind="bp", Lx=5, Ly=5, chi=32, prec="fp32", sweeps=10),
        # measuring a stored state again
        dict(name="measure_4x4_chi64_tf32x3", kind="measure", Lx=4, Ly=4, chi=64, prec="tf32x3", sweeps=10),
        # one training step of the warm start on the rows of one 10x10, chi = 100 layer
        dict(name="train_36000", kind="train", rows=36000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evolve", "layer", "layer", "layer", "bp", "bp", "measure", "train"])
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 400, 36000))
    if kind == "evolve":
        n = rng.choice([1, 1, rng.randint(2, 9)])
        prec = rng.choice(["fp64", "fp32", "tf32x3"])
        return dict(kind=kind, Lx=rng.randint(2, 4), Ly=rng.randint(3, 5), chi=_log_int(rng, 6, 14 if prec == "fp64" else 20),
                    prec=prec, order=rng.choice([1, 2]), steps=rng.randint(3, 5), sweeps=rng.randint(20, 26) if prec == "fp64" else rng.randint(16, 20), n=n)
    prec = rng.choice(["fp64", "fp32", "fp32", "tf32x3", "tf32x3", "tf32x3"])
    top = {"fp64": 14, "fp32": 44, "tf32x3": 90}[prec]
    chi = _log_int(rng, 7, top)
    Lx, Ly = rng.randint(2, 4), rng.randint(3, 5)
    if chi > 32:
        Lx, Ly = rng.randint(2, 3), rng.randint(3, 4)
    if chi > 64:
        Ly = 3
    c = dict(kind=kind, Lx=Lx, Ly=Ly, chi=chi, prec=prec, sweeps=rng.randint(3, 12))
    if kind == "layer":
        c.update(order=rng.choice([1, 2]), sweeps=rng.randint(24, 28) if prec == "fp64" else rng.randint(16, 20))
    return c


# ------------------------------------------------------------------ inputs
def _grid(Lx, Ly):
    """Bonds (first site, second site, colour) in the library's order and, per site,
    its (bond, neighbour) legs in the order up, down, left, right."""
    bonds = [(y * Lx + x, y * Lx + x + 1, x % 2) for y in range(Ly) for x in range(Lx - 1)]
    bonds += [(y * Lx + x, (y + 1) * Lx + x, 2 + y % 2) for y in range(Ly - 1) for x in range(Lx)]
    ident = {(a, b): i for i, (a, b, _) in enumerate(bonds)}
    legs = []
    for v in range(Lx * Ly):
        x, y = v % Lx, v // Lx
        around = [(x, y - 1), (x, y + 1), (x - 1, y), (x + 1, y)]
        there = [q * Lx + p for p, q in around if 0 <= p < Lx and 0 <= q < Ly]
        legs.append([(ident[min(v, w), max(v, w)], w) for w in there])
    return bonds, legs


def _sizes(case):
    """(Lx, Ly, chi) of every instance of a case."""
    if case.get("n", 1) == 1:
        return [(case["Lx"], case["Ly"], case["chi"])]
    return [(case["Lx"] + i % 3, case["Ly"] + i % 3, case["chi"] * (1 + i // 3 % 3)) for i in range(case["n"])]


def _configs(case, seed):
    rng = random.Random(int(seed))
    got = []
    for Lx, Ly, chi in _sizes(case):
        h = rng.uniform(0.5, 3.0) if case["kind"] == "evolve" else 2.0
        got.append(dict(Lx=Lx, Ly=Ly, J=1.0, h=h, dt=0.05, order=case.get("order", 2), obs=((Lx - 1) // 2, (Ly - 1) // 2),
                        chi_max=chi, eps_cut=EPS_CUT, bp_alpha=0.5, bp_tol=OUT_OF_REACH, bp_max_sweeps=case["sweeps"],
                        qr_ratio_thresh=16.0 if case["prec"] == "tf32x3" else 150.0, precision=case["prec"]))
    return got


def _spectrum(chi):
    lam = np.exp(-DECAY * np.arange(chi))
    return lam / np.linalg.norm(lam)


def _site(cfg, legs, seed, v):
    """A seeded site tensor: Gaussian entries, each leg weighted by the square root of
    its spectrum; the Pauli component that the correlator pins is half-normal, so that
    single-layer BP meets the positive network that evolved operators give it."""
    dtype = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    chi, d = cfg["chi_max"], len(legs[v])
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 4099 + v)
    t = torch.randn((chi,) * d + (4,), generator=gen, device="cuda", dtype=dtype)
    pin = 3 if v == cfg["obs"][1] * cfg["Lx"] + cfg["obs"][0] else 0
    t[..., pin].abs_()
    root = torch.as_tensor(np.sqrt(_spectrum(chi)), device="cuda", dtype=dtype)
    for k in range(d):
        t *= root.reshape((chi,) + (1,) * (d - k))
    t *= torch.tensor(WEIGHT, device="cuda", dtype=dtype)
    return t


def _network(seed):
    """Weights of the warm-start network, He-scaled, and its training rows."""
    rng = np.random.default_rng(int(seed))
    p = dict(W1=rng.standard_normal((12, 256)) * math.sqrt(2 / 12), b1=rng.standard_normal(256) * 0.1,
             W2=rng.standard_normal((256, 256)) * math.sqrt(2 / 256), b2=rng.standard_normal(256) * 0.1,
             W3=rng.standard_normal((256, 1)) * math.sqrt(1 / 256), b3=rng.standard_normal(1) * 0.1)
    return {k: v.astype(np.float32) for k, v in p.items()}


def _rows(case, seed):
    """Feature rows as a layer gives them (log spectra, fractions, distances) and targets."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 31 + 7)
    u = torch.rand((case["rows"], 12), generator=gen, device="cuda")
    scale = torch.tensor([-7.0, 1, 0.8, 1, 1, 1, 1, 2, 2.5, 1, 0.8, 0.9], device="cuda")
    X = u * scale
    t = 2.0 * X[:, 0] - 1.0 + 0.3 * torch.randn(case["rows"], generator=gen, device="cuda")
    return X.contiguous(), t.contiguous()


def prepare(case, seed):
    if case["kind"] == "train":
        X, t = _rows(case, seed)
        return dict(kind="train", mlp=pkg.Mlp(pkg.flat_params(_network(seed)), case["rows"]), X=X, t=t)
    cfgs = _configs(case, seed)
    eng = pkg.Engine([pkg.Config(**c) for c in cfgs])
    if case["kind"] != "evolve":
        c = cfgs[0]
        bonds, legs = _grid(c["Lx"], c["Ly"])
        lam = _spectrum(c["chi_max"])
        eng.set_bonds(0, np.full(len(bonds), c["chi_max"]), np.tile(lam, (len(bonds), 1)), np.tile(np.diag(lam), (len(bonds), 2, 1, 1)))
        for v in range(len(legs)):
            eng.set_site(0, v, _site(c, legs, seed, v).cpu().numpy())
    snaps = [torch.empty(eng.state_bytes(i), dtype=torch.uint8, device="cuda") for i in range(len(cfgs))]
    for i, s in enumerate(snaps):
        eng.save_state(s, i)
    return dict(kind=case["kind"], eng=eng, snaps=snaps, cfgs=cfgs, steps=case.get("steps", 0),
                dtype=np.float64 if case["prec"] == "fp64" else np.float32)


# -------------------------------------------------------------------- one pass
def _spectra(eng, i, c):
    out = np.zeros((eng.num_bonds(i), c["chi_max"]))
    for b in range(len(out)):
        lam = eng.spectrum(i, b)
        out[b, : len(lam)] = lam
    return out


def _scalars(d):
    return [d["C"], d["C_proj"], d["log_norm"], d["gate_err"]]


def run(state):
    if state["kind"] == "train":
        loss, grad = state["mlp"].gradient(state["X"], state["t"], want_grad=True)
        state["mlp"].adam_step(1e-3)
        return dict(loss=loss, grad=grad, params=state["mlp"].params())
    eng, cfgs, dtype = state["eng"], state["cfgs"], state["dtype"]
    for i, s in enumerate(state["snaps"]):
        eng.load_state(s, i)
    if state["kind"] == "bp":
        eng.bp_converge()
        return dict(messages=eng.get_messages(0).astype(dtype))
    if state["kind"] == "measure":
        D = [eng.correlator()[1]]
    elif state["kind"] == "layer":
        eng.trotter_step(1)
        eng.bp_converge()
        D = [eng.correlator()[1]]
    else:
        D = eng.run(state["steps"])
        D = [d if isinstance(d, list) else [d] for d in D]
    out = dict(measured=np.array([[_scalars(d) for d in row] for row in D]).astype(dtype),
               pauli=np.concatenate([eng.pauli_weights(i).ravel() for i in range(len(cfgs))]).astype(dtype))
    if state["kind"] != "measure":
        out["spectra"] = np.concatenate([_spectra(eng, i, c).ravel() for i, c in enumerate(cfgs)]).astype(dtype)
    return out


# ------------------------------------------------------------------ what it takes
def _work_instance(Lx, Ly, chi_of, case, item):
    """Bytes and operations of one layer (and its BP sweeps) at bond dimension chi_of."""
    _, legs = _grid(Lx, Ly)
    by = fl = 0.0
    for l in legs:
        d, chi = len(l), chi_of
        size = 4.0 * chi ** d
        if case["kind"] in ("layer", "evolve"):
            n, m = 4.0 * chi, size / (4.0 * chi)
            # per update: absorb the other legs, one Gram or QR, the new tensor
            fl += d * (2.0 * chi * size * (d - 1) + m * n * n + 2.0 * m * n * n)
            by += 2.0 * size * item
        if case["kind"] in ("layer", "evolve", "bp"):
            # per sweep: rotate every leg, one symmetric Gram per leg
            fl += case["sweeps"] * d * (2.0 * chi * size + chi * size)
        if case["kind"] != "bp":
            # single-layer sweeps on the pinned slice, the closing double-layer pass
            fl += (case["sweeps"] + 1) * 4.0 * size / 4.0 + d * 2.0 * chi * size + chi * size
        if case["kind"] in ("bp", "measure"):
            by += size * item
        by += 8.0 * chi * chi * d * (2 if case["kind"] == "bp" else 1)
    return by, fl


def work(case):
    if case["kind"] == "train":
        n = 12 * 256 + 256 + 256 * 256 + 256 + 256 + 1
        return dict(bytes=4.0 * (13 * case["rows"] + 7 * n), flops=6.0 * case["rows"] * (12 * 256 + 256 * 256 + 256))
    item = 8 if case["prec"] == "fp64" else 4
    by = fl = 0.0
    for Lx, Ly, chi in _sizes(case):
        if case["kind"] == "evolve":
            # bonds grow from 1, about twofold a step, up to chi_max
            for s in range(1, case["steps"] + 1):
                b, f = _work_instance(Lx, Ly, min(chi, 2 ** s), case, item)
                by, fl = by + b, fl + f
        else:
            by, fl = _work_instance(Lx, Ly, chi, case, item)
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------- the same in 64 bits, plainly
_PAULI = [np.eye(2), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1.0, -1.0])]


def _transfer(g, ops):
    """T[a, b] = Re Tr(P_a g^dagger P_b g) / dim."""
    return np.array([[np.trace(a @ g.conj().T @ b @ g).real / len(g) for b in ops] for a in ops])


def _leg(A, T, k):
    """T with A (rows x leg) applied to leg k."""
    return torch.movedim(torch.tensordot(A, T, dims=([1], [k])), 0, k)


class _Net:
    """The method of the paper in 64 bits: messages of bond b in direction 0 (first site
    to second) and 1 are M[2 b] and M[2 b + 1]."""

    def __init__(self, cfg, dev):
        self.c, self.dev = cfg, dev
        self.bonds, self.legs = _grid(cfg["Lx"], cfg["Ly"])
        self.pin = [0] * len(self.legs)
        self.pin[cfg["obs"][1] * cfg["Lx"] + cfg["obs"][0]] = 3
        self.gate_err = 0.0
        Z, X = _PAULI[3], _PAULI[1]
        th = cfg["J"] * cfg["dt"]
        ph = cfg["h"] * cfg["dt"] * (0.5 if cfg["order"] == 2 else 1.0)
        two = [np.kron(a, b) for a in _PAULI for b in _PAULI]
        G = _transfer(np.cos(th) * np.eye(4) - 1j * np.sin(th) * np.kron(Z, Z), two)
        self.S = self._t(_transfer(np.cos(ph) * np.eye(2) - 1j * np.sin(ph) * X, _PAULI))
        # operator-Schmidt factors: G[(a1 a2), (b1 b2)] = sum_k F1[k, a1, b1] F2[k, a2, b2]
        u, s, vt = np.linalg.svd(G.reshape(4, 4, 4, 4).transpose(0, 2, 1, 3).reshape(16, 16))
        r = int(np.sum(s > 1e-12 * s[0]))
        self.F = [self._t((u[:, :r] * np.sqrt(s[:r])).T.reshape(r, 4, 4)), self._t((vt[:r].T * np.sqrt(s[:r])).T.reshape(r, 4, 4))]

    def _t(self, x):
        return torch.as_tensor(np.asarray(x), dtype=torch.float64, device=self.dev)

    def initial(self):
        self.T = []
        for v, l in enumerate(self.legs):
            e = torch.zeros(4, dtype=torch.float64, device=self.dev)
            e[self.pin[v]] = 1.0
            self.T.append(e.reshape((1,) * len(l) + (4,)))
        self.lam = [self._t([1.0]) for _ in self.bonds]
        self.M = [self._t([[1.0]]) for _ in range(2 * len(self.bonds))]
        return self

    def saturated(self, seed):
        lam = self._t(_spectrum(self.c["chi_max"]))
        self.T = [_site(self.c, self.legs, seed, v).to(self.dev).double() for v in range(len(self.legs))]
        self.lam = [lam for _ in self.bonds]
        self.M = [torch.diag(lam) for _ in range(2 * len(self.bonds))]
        return self

    def into(self, v, b):
        return 2 * b if self.bonds[b][1] == v else 2 * b + 1

    def out_of(self, v, b):
        return 2 * b if self.bonds[b][0] == v else 2 * b + 1

    def update(self, b):
        side = []
        for i in (0, 1):
            v = self.bonds[b][i]
            cut = [x[0] for x in self.legs[v]].index(b)
            T = self.T[v]
            back = []
            for k, (e, _) in enumerate(self.legs[v]):
                if k == cut:
                    continue
                M = self.M[self.into(v, e)]
                d, V = torch.linalg.eigh(0.5 * (M + M.T))
                keep = d > 1e-12 * d[-1]
                root = d[keep].sqrt()
                T = _leg(root[:, None] * V[:, keep].T, T, k)
                back.append((k, V[:, keep] / root))
            T = torch.movedim(T, cut, -2)
            env, chi = T.shape[:-2], T.shape[-2]
            Q, R = torch.linalg.qr(T.reshape(-1, chi * 4))
            X = torch.einsum("kab,rcb->rack", self.F[i], R.reshape(-1, chi, 4))
            K = X.shape[0]
            q, t = torch.linalg.qr(X.reshape(K * 4, -1))
            side.append((v, cut, back, env, Q, q, t, K))
        U, s, Vt = torch.linalg.svd(side[0][6] @ side[1][6].T, full_matrices=False)
        n = min(self.c["chi_max"], max(1, int((s >= EPS_CUT * s[0]).sum())))
        tot, kept = float((s * s).sum()), float((s[:n] * s[:n]).sum())
        self.gate_err += (tot - kept) / tot
        root = s[:n].sqrt()
        for (v, cut, back, env, Q, q, _, K), W in zip(side, (U[:, :n], Vt[:n].T)):
            Y = (q @ (W * root)).reshape(K, 4 * n)
            T = (Q @ Y).reshape(env + (4, n))
            T = torch.movedim(T, -1, cut)
            for k, A in back:
                T = _leg(A, T, k)
            self.T[v] = T
        self.lam[b] = s[:n] / math.sqrt(kept)
        self.M[2 * b] = self.M[2 * b + 1] = torch.diag(self.lam[b])

    def site_gates(self):
        self.T = [T @ self.S.T for T in self.T]

    def step(self):
        self.gate_err = 0.0
        self.site_gates()
        for colour in range(4):
            for b, (_, _, c) in enumerate(self.bonds):
                if c == colour:
                    self.update(b)
        if self.c["order"] == 2:
            self.site_gates()

    def hats(self):
        """Unnormalised outgoing messages of every site."""
        got = [None] * len(self.M)

        def rest(v, T, todo):
            if len(todo) == 1:
                k = todo[0]
                A = torch.movedim(T, k, 0).reshape(T.shape[k], -1)
                B = torch.movedim(self.T[v], k, 0).reshape(T.shape[k], -1)
                got[self.out_of(v, self.legs[v][k][0])] = B @ A.T
                return
            half = len(todo) // 2
            for keep, drop in ((todo[:half], todo[half:]), (todo[half:], todo[:half])):
                U = T
                for k in drop:
                    U = _leg(self.M[self.into(v, self.legs[v][k][0])], U, k)
                rest(v, U, keep)

        for v, l in enumerate(self.legs):
            rest(v, self.T[v], list(range(len(l))))
        return got

    def bp(self):
        for _ in range(self.c["bp_max_sweeps"]):
            H = self.hats()
            a = self.c["bp_alpha"]
            self.M = [(1 - a) * M + a * 0.5 * (h + h.T) / torch.trace(h) for M, h in zip(self.M, H)]

    def vhats(self, vec):
        got = [None] * len(self.M)
        for v, l in enumerate(self.legs):
            for w in range(len(l)):
                T = self.T[v][..., self.pin[v]]
                for k in reversed(range(len(l))):
                    if k != w:
                        T = torch.tensordot(T, vec[self.into(v, l[k][0])], dims=([k], [0]))
                got[self.out_of(v, l[w][0])] = T
        return got

    def measure(self):
        vec = []
        for M in self.M:
            m = torch.diagonal(M).clamp(min=0).sqrt()
            vec.append(m / m.norm())
        a = self.c["bp_alpha"]
        for _ in range(self.c["bp_max_sweeps"]):
            new = []
            for h, m in zip(self.vhats(vec), vec):
                h = h / h.norm()
                new.append((1 - a) * m + a * (h if float(h @ m) >= 0 else -h))
            vec = new
        H, h = self.hats(), self.vhats(vec)
        lc = ln = 0.0
        sign = 1.0
        for v, l in enumerate(self.legs):
            o, i = self.out_of(v, l[-1][0]), self.into(v, l[-1][0])
            x = float(h[o] @ vec[i])
            sign = -sign if x < 0 else sign
            lc += math.log(abs(x))
            ln += math.log(float((H[o] * self.M[i]).sum()))
        for b in range(len(self.bonds)):
            z = float(vec[2 * b] @ vec[2 * b + 1])
            sign = -sign if z < 0 else sign
            lc -= math.log(abs(z))
            ln -= math.log(float((self.M[2 * b] * self.M[2 * b + 1]).sum()))
        return [sign * math.exp(lc - 0.5 * ln), sign * math.exp(lc), ln, self.gate_err]

    def pauli(self):
        out = []
        for v, l in enumerate(self.legs):
            T = self.T[v]
            for k, (e, _) in enumerate(l):
                T = _leg(self.M[self.into(v, e)], T, k)
            w = (T * self.T[v]).reshape(-1, 4).sum(0)
            out.append(w / w.sum())
        return torch.cat(out).cpu().numpy()

    def spectra(self):
        out = np.zeros((len(self.bonds), self.c["chi_max"]))
        for b, lam in enumerate(self.lam):
            out[b, : len(lam)] = lam.cpu().numpy()
        return out.ravel()


def _bf16(x):
    return x.float().bfloat16().double()


def _exact_train(case, seed):
    """The network with its weights and activations rounded to BF16 where the framework
    says that they are; every sum in 64 bits."""
    X, t = (x.double() for x in _rows(case, seed))
    p = {k: torch.as_tensor(v, device="cuda").double() for k, v in _network(seed).items()}
    gelu = lambda z: 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))  # noqa: E731
    slope = lambda z: 0.5 * (1 + torch.erf(z / math.sqrt(2))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)  # noqa: E731
    x, W1, W2, W3 = _bf16(X), _bf16(p["W1"]), _bf16(p["W2"]), _bf16(p["W3"])
    z1 = x @ W1 + p["b1"]
    a1 = _bf16(gelu(z1))
    z2 = a1 @ W2 + p["b2"]
    a2 = _bf16(gelu(z2))
    y = (a2 @ W3)[:, 0] + p["b3"]
    dy = 2 * (y - t) / len(t)
    d2 = dy[:, None] * W3[:, 0] * slope(z2)
    d1 = (d2 @ W2.T) * slope(z1)
    grad = torch.cat([(x.T @ d1).ravel(), d1.sum(0), (a1.T @ d2).ravel(), d2.sum(0), a2.T @ dy, dy.sum().reshape(1)])
    flat = torch.cat([p[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")])
    return dict(loss=float(((y - t) ** 2).mean()), grad=grad.cpu().numpy(), params=(flat - 1e-3 * grad / (grad.abs() + 1e-8)).cpu().numpy())


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    nets, rows = [], []
    for cfg in _configs(case, seed):
        small = 4 * cfg["chi_max"] ** 4 <= 10 ** 6 or case["kind"] == "evolve"
        net = _Net(cfg, "cpu" if small else "cuda")
        nets.append(net.initial() if case["kind"] == "evolve" else net.saturated(seed))
    if case["kind"] == "bp":
        nets[0].bp()
        return dict(messages=torch.stack(nets[0].M).cpu().numpy())
    if case["kind"] == "layer":
        nets[0].step()
        nets[0].bp()
    if case["kind"] == "evolve":
        for net in nets:
            net.bp()
            got = [net.measure()]
            for _ in range(case["steps"]):
                net.step()
                net.bp()
                got.append(net.measure())
            rows.append(got)
        measured = np.array(rows).transpose(1, 0, 2)
    else:
        measured = np.array([[nets[0].measure()]])
    out = dict(measured=measured, pauli=np.concatenate([n.pauli() for n in nets]))
    if case["kind"] != "measure":
        out["spectra"] = np.concatenate([n.spectra() for n in nets])
    return out
