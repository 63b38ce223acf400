"""The work that users of the TU-fRG library have it do, as measurable cases.

Most calls are right-hand sides: an adaptive flow evaluates nothing else, and callers with integrators of their own call
``Model.rhs`` directly.  The cases cover both precisions, states with the lattice symmetries (every state of a flow) and
general ones, one- and many-orbital models, and the meshes and bond sets of the library's workloads; one whole flow and
one training step of the loop surrogate stand beside them.

The split path returns values that are FP32 by construction, widened to the complex128 of the state's layout.  Its
callers keep them in the precision they have (half the memory), and so do these cases: the pass ends with the copy into a
complex64 buffer.  The FP64 path's results are kept as they are.
"""
import math

import numpy as np
import torch

from paper_1710_08830_gb300 import inputs
from paper_1710_08830_gb300.api import CH_C, CH_P, FP64, SPLIT32, Model
from paper_1710_08830_gb300.surrogate import Net

SHELL_T = 0.05   # temperature of the momentum-shell regulator's Fermi functions


def _rhs(name, family, Lq, nc, n_ff, split, symmetric, T, shell=False):
    return dict(name=name, kind="rhs", family=family, Lq=Lq, nc=nc, n_ff=n_ff, split=split, symmetric=symmetric, T=T,
                shell=shell)


def listed():
    return [
        # the smallest flow in use (one band, coarse mesh, M = 20): a stage of it is a chain of launches of a few us
        _rhs("hubbard_q8_split", "hubbard", 8, 16, 5, True, True, 0.1),
        # the benchmark's workload, a stage of a mid-flow step
        _rhs("rashba_q24_split", "rashba", 24, 8, 9, True, True, 0.1),
        # the same model on a state without the lattice symmetries (a perturbed or symmetry-broken start)
        _rhs("rashba_q24_split_general", "rashba", 24, 8, 9, True, False, 0.1),
        # the largest members of the batched flows: 48 x 48 momenta, 13 bonds (M = 52), late in the flow
        _rhs("rashba_q48_ff13_split", "rashba", 48, 8, 13, True, True, 0.05),
        # plain FP64 twins of the first two: reference flows, and the accuracy statements of the split path
        _rhs("hubbard_q8_fp64", "hubbard", 8, 16, 5, False, True, 0.1),
        _rhs("rashba_q24_fp64", "rashba", 24, 8, 9, False, False, 0.1),
        # three-orbital model with spin-orbit coupling (M = 324), the largest state (3.4 GB)
        _rhs("t2g_q32_split", "t2g", 32, 6, 9, True, True, 0.1),
        # the same family on an odd mesh and a general state: every momentum projected and multiplied
        _rhs("t2g_q15_split_general", "t2g", 15, 6, 9, True, False, 0.3),
        # its FP64 path on a mesh where a reference flow is affordable
        _rhs("t2g_q8_fp64", "t2g", 8, 6, 9, False, True, 0.1),
        # two layers (N_s = 4) on an odd fine mesh
        _rhs("bilayer_q12_split", "bilayer", 12, 5, 9, True, True, 0.2),
        # a whole flow through the public call: about 60 attempts of six right-hand sides, error norms and commits
        dict(name="hubbard_flow_split", kind="flow", family="hubbard", Lq=8, nc=16, n_ff=5, split=True, T_end=0.02),
        # one training step's gradients of the loop surrogate at its batch size
        dict(name="surrogate_gradients_b1024", kind="mlp", batch=1024, width=256, depth=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs2", "rhs2", "rhs2", "rhs2_64", "rhs2_64", "t2g", "t2g_64", "bilayer", "flow", "mlp"])
    T = round(math.exp(rng.uniform(math.log(0.02), math.log(10.0))), 4)
    shell, symmetric = rng.random() < 0.2, rng.random() < 0.5
    if kind in ("rhs2", "rhs2_64"):
        split = kind == "rhs2"
        Lq = _log_int(rng, 5, 48 if split else 24)
        nc = rng.randint(2, max(2, min(16, (384 if split else 192) // Lq)))
        c = _rhs("", rng.choice(["hubbard", "rashba"]), Lq, nc, rng.choice([5, 9, 13]), split, symmetric, T, shell)
    elif kind == "t2g":
        c = _rhs("", "t2g", rng.randint(4, 24), rng.randint(2, 6), rng.choice([5, 9]), True, symmetric, T, shell)
    elif kind == "t2g_64":
        c = _rhs("", "t2g", rng.randint(4, 8), rng.randint(2, 6), rng.choice([5, 9]), False, symmetric, T, shell)
    elif kind == "bilayer":
        c = _rhs("", "bilayer", rng.randint(5, 16), rng.randint(2, 6), rng.choice([5, 9, 13]), rng.random() < 0.7,
                 symmetric, T, shell)
    elif kind == "flow":
        c = dict(kind="flow", family=rng.choice(["hubbard", "rashba"]), Lq=rng.randint(5, 12), nc=rng.randint(4, 16),
                 n_ff=rng.choice([5, 9]), split=True, T_end=round(math.exp(rng.uniform(math.log(0.02), 0.0)), 4))
    else:
        c = dict(kind="mlp", batch=_log_int(rng, 64, 4096), width=rng.choice([128, 200, 256]), depth=rng.randint(2, 4))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------------ inputs
def _spec(c, seed):
    kw = dict(Lq=c["Lq"], nc=c["nc"], n_ff=c["n_ff"])
    if c["kind"] == "flow":   # a flow's inputs are its model: the interaction and t' of this seed
        r = np.random.default_rng(seed)
        U, tp = float(r.uniform(2.0, 3.0)), float(r.uniform(-0.3, -0.1))
    else:
        U, tp = None, None
    if c["family"] == "hubbard":
        spec = inputs.hubbard_square(1.0, -0.25 if tp is None else tp, 3.0 if U is None else U, filling=0.9, **kw)
    elif c["family"] == "rashba":
        spec = inputs.rashba_hubbard(1.0, -0.2 if tp is None else tp, 0.3, 2.5 if U is None else U, -0.818, **kw)
    elif c["family"] == "bilayer":
        spec = inputs.rashba_bilayer(**kw)
    else:
        spec = inputs.t2g_soc(0, 0.2, 2.0, 0.4, filling=4.0, **kw)
    return spec.with_(regulator=1, T_reg=SHELL_T) if c.get("shell") else spec


def _pair_matrices(spec, dev):
    """The bare vertex as a matrix over orbital pairs: P rows (s1,s2), columns (s4,s3); C rows (s1,s3), columns (s4,s2)."""
    n2 = spec.n_s ** 2
    V = torch.from_numpy(np.ascontiguousarray(spec.V0)).to(dev)
    return V.permute(0, 1, 3, 2).reshape(n2, n2), V.permute(0, 2, 3, 1).reshape(n2, n2)


_POINT = [(1, 0, 0, 1), (0, -1, 1, 0), (-1, 0, 0, -1), (0, 1, -1, 0), (-1, 0, 0, 1), (1, 0, 0, -1), (0, 1, 1, 0), (0, -1, -1, 0)]


def _symmetric_state(spec, seed, dev):
    """A state with the symmetries of the square lattice and of the interaction: random bond matrices averaged over the
    point group and q -> -q, times the unit matrix and the bare vertex over the orbital pairs."""
    g = torch.Generator(device=dev).manual_seed(seed)
    F, L, n2 = spec.n_ff, spec.Lq, spec.n_s ** 2
    bonds = [tuple(int(x) for x in b) for b in spec.ff_R]
    x, y = torch.meshgrid(torch.arange(L, device=dev), torch.arange(L, device=dev), indexing="ij")
    X = torch.empty((2, spec.Nq, F, n2, F, n2), dtype=torch.complex128, device=dev)
    for ch, V in enumerate(_pair_matrices(spec, dev)):
        X[ch] = 0
        for K, scale in ((torch.eye(n2, dtype=torch.complex128, device=dev), 0.2), (V, 0.2)):
            a = torch.randn((spec.Nq, F, F), dtype=torch.float64, device=dev, generator=g)
            a = a + a.transpose(1, 2)
            s = torch.zeros_like(a)
            for G in _POINT:
                perm = torch.tensor([bonds.index((G[0] * b[0] + G[1] * b[1], G[2] * b[0] + G[3] * b[1])) for b in bonds], device=dev)
                for sign in (1, -1):   # time reversal: q -> -q at the same bonds
                    q = (sign * (G[0] * x + G[1] * y) % L * L + sign * (G[2] * x + G[3] * y) % L).reshape(-1)
                    s += a[q][:, perm][:, :, perm]
            s *= scale / 16
            X[ch] += torch.einsum("qij,ab->qiajb", s.to(torch.complex128), K)
    return X.reshape(2, spec.Nq, F * n2, F * n2)


def _general_state(spec, seed, dev):
    """Hermitian per momentum, no other symmetry."""
    g = torch.Generator(device=dev).manual_seed(seed)
    X = torch.randn((2, spec.Nq, spec.M, spec.M), dtype=torch.complex128, device=dev, generator=g) * 0.3
    return (0.5 * (X + X.mH)).contiguous()


def _state(c, spec, seed, dev):
    return _symmetric_state(spec, seed, dev) if c["symmetric"] else _general_state(spec, seed, dev)


def _net(c, seed):
    """(flat parameters, features, targets) of a training batch: He-uniform weights, the features of random momenta
    and model parameters, standardised targets."""
    r = np.random.default_rng(seed)
    dims = [20] + [c["width"]] * c["depth"] + [1600]
    p = []
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        s = math.sqrt(6.0 / a) * (0.5 if i == len(dims) - 2 else 1.0)
        p += [r.uniform(-s, s, a * b), r.uniform(-0.1, 0.1, b)]
    q = 2 * math.pi * r.integers(0, 24, (c["batch"], 2)) / 24
    n = np.arange(1, 5)[None, :]
    wave = [np.sin(n * q[:, :1]), np.cos(n * q[:, :1]), np.sin(n * q[:, 1:]), np.cos(n * q[:, 1:])]
    X = np.concatenate([np.stack(wave, 2).reshape(c["batch"], 16), r.uniform(-1, 1, (c["batch"], 4))], 1)
    return np.concatenate(p).astype(np.float32), X.astype(np.float32), r.standard_normal((c["batch"], 1600)).astype(np.float32)


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["kind"] == "mlp":
        p, X, Y = _net(case, seed)
        net = Net(20, case["width"], case["depth"], 1600)
        net.set_params(p)
        return dict(net=net, X=torch.from_numpy(X).to(dev), Y=torch.from_numpy(Y).to(dev))
    spec = _spec(case, seed)
    model = Model(spec, SPLIT32 if case["split"] else FP64)
    if case["kind"] == "flow":
        return dict(case=case, model=model)
    out = model.zeros_state()
    return dict(case=case, model=model, X=_state(case, spec, seed, dev), out=out,
                kept=torch.empty_like(out, dtype=torch.complex64) if case["split"] else None)


def run(state):
    if "net" in state:
        loss, g = state["net"].gradients(state["X"], state["Y"])
        return {"loss": loss, "grad": g}
    c, m = state["case"], state["model"]
    if c["kind"] == "flow":
        X, r = m.flow(T_end=c["T_end"])
        return {"state": X.to(torch.complex64), "Tc": r["Tc"], "amax": r["amax"]}
    m.rhs(c["T"], state["X"], mask=CH_P | CH_C, out=state["out"], symmetric=c["symmetric"])
    return state["out"] if state["kept"] is None else state["kept"].copy_(state["out"])


# ------------------------------------------------------------------------------------------ work
def _orbits(L):
    h = L // 2 + 1
    return h * (h + 1) // 2


def work(case):
    """A right-hand side reads the state and writes the derivative; its loops are, per orbit of transfer momenta, channel and
    point of half the fine mesh (the other half follows by exchange of the two propagators), N_s^5 multiply-adds for the
    weighted projectors' product and 2 n_dy - 1 real row phases of its N_s^4 entries; its products two complex M^3."""
    if case["kind"] == "mlp":
        dims = [20] + [case["width"]] * case["depth"] + [1600]
        n = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
        return {"bytes": 4.0 * (2 * n + case["batch"] * 1620), "flops": 6.0 * n * case["batch"]}
    ns = {"hubbard": 2, "rashba": 2, "bilayer": 4, "t2g": 6}[case["family"]]
    Nq, M, reps = case["Lq"] ** 2, case["n_ff"] * ns * ns, _orbits(case["Lq"])
    ndy = {1: 1, 5: 3, 9: 3, 13: 5}[case["n_ff"]]
    symmetric = case.get("symmetric", True)
    loops = 2.0 * 2 * reps * (Nq * case["nc"] ** 2 / 2) * (ns ** 5 + (2 * ndy - 1) * ns ** 4)
    prods = 2.0 * 2 * 8 * M ** 3 * (reps if symmetric else Nq)
    per = {"bytes": 2.0 * 16 * 2 * Nq * M * M, "flops": loops + prods}
    if case["kind"] == "flow":   # at least 40 accepted steps of six evaluations on the way to T_end = 0.02
        n = 6 * max(4, int(40 * math.log(10.0 / case["T_end"]) / math.log(500.0)))
        return {k: v * n for k, v in per.items()}
    return per


# ------------------------------------------------------------------------------------------ the same in 64 bits
def _bands(spec):
    k = 2 * np.pi * np.arange(spec.Lf) / spec.Lf
    ph = np.exp(1j * (k[:, None, None] * spec.hop_R[:, 0] + k[None, :, None] * spec.hop_R[:, 1])).reshape(spec.Nk, -1)
    E, U = np.linalg.eigh(np.einsum("kr,rab->kab", ph, spec.hop_t))
    mu = spec.mu
    if spec.filling > 0:
        lo, hi = E.min() - 1.0, E.max() + 1.0
        for _ in range(200):
            mu = 0.5 * (lo + hi)
            n = float(np.sum(0.5 * (1.0 - np.tanh(0.5 * (E - mu) / spec.T_mu)))) / spec.Nk
            lo, hi = (mu, hi) if n < spec.filling else (lo, mu)
    return E - mu, U


def _weights(which, shell, T, e, fd, i1, i2):
    """Loop weights of every band pair of the points i1, i2; fd = (g, g') of the temperature flow, (f, h) of the shell."""
    a, b = e[i1][:, :, None], e[i2][:, None, :]
    u1, v1, u2, v2 = fd[0][i1][:, :, None], fd[1][i1][:, :, None], fd[0][i2][:, None, :], fd[1][i2][:, None, :]
    den = a + b if which == 0 else a - b
    near = den.abs() <= 1e-5 * (SHELL_T if shell else T)
    den = torch.where(near, torch.ones_like(den), den)
    if not shell:
        return torch.where(near, (-0.5 if which == 0 else 0.5) * (v1 + v2), (-(u1 + u2) if which == 0 else u1 - u2) / den)
    F = torch.where(near, (0.5 if which == 0 else -0.5) * (v1 + v2), ((1 - u1 - u2) if which == 0 else u1 - u2) / den)
    q1, q2 = a * a + T * T, b * b + T * T
    return -2 * T * a * a * b * b * (q1 + q2) / (q1 * q2) ** 2 * F


def _loops(spec, T, shell, dev):
    """[channel][q][bond difference][pair][pair] by the direct k-sum, and the sorted differences."""
    L, Lf, nc, ns = spec.Lq, spec.Lf, spec.nc, spec.n_s
    n2 = ns * ns
    E, U = _bands(spec)
    e, U = torch.from_numpy(E).to(dev), torch.from_numpy(U).to(dev)
    Tf = SHELL_T if shell else T
    x = (e.abs() / Tf)
    z = torch.exp(-x)
    if shell:
        fd = (torch.where(e > 0, z / (1 + z), 1 / (1 + z)), z / (1 + z) ** 2 / Tf)
    else:
        h = z / (1 + z) ** 2
        fd = (e / T / T * h, h / T ** 2 * (1 - x * (1 - z) / (1 + z)))
    rho = torch.einsum("ktl,kul->kltu", U, U.conj()).reshape(-1, ns, n2)
    d = sorted({(int(a[0] - b[0]), int(a[1] - b[1])) for a in spec.ff_R for b in spec.ff_R})
    half = [v for v in d if v[1] > 0 or (v[1] == 0 and v[0] >= 0)]
    kx, ky = torch.meshgrid(torch.arange(Lf, device=dev), torch.arange(Lf, device=dev), indexing="ij")
    kx, ky = kx.reshape(-1), ky.reshape(-1)
    D = torch.tensor(half, device=dev)
    ang = (kx[None] * D[:, :1] + ky[None] * D[:, 1:]) % Lf
    ph = torch.polar(torch.ones(ang.shape, dtype=torch.float64, device=dev), -2 * math.pi * ang.double() / Lf) / spec.Nk
    out = torch.empty((2, spec.Nq, len(d), n2, n2), dtype=torch.complex128, device=dev)
    for ch in (0, 1):
        for q in range(spec.Nq):
            sx, sy = q // L * nc, q % L * nc
            if ch == 0:
                i1, i2 = (sx - kx) % Lf * Lf + (sy - ky) % Lf, kx * Lf + ky
                r2 = rho
            else:
                i1, i2 = kx * Lf + ky, (kx - sx) % Lf * Lf + (ky - sy) % Lf
                r2 = rho.conj()
            w = _weights(ch, shell, T, e, fd, i1, i2)
            t = torch.einsum("kij,kjb->kib", w.to(torch.complex128), r2[i2])
            y = torch.bmm(rho[i1].transpose(1, 2), t).reshape(-1, n2 * n2)
            lc = (ph @ y).reshape(len(half), ns, ns, ns, ns)          # [t1][t3][t2][t4]
            lc = lc.permute(0, 3, 1, 4, 2) if ch == 0 else lc.permute(0, 1, 3, 2, 4)
            lc = lc.reshape(len(half), n2, n2)
            for i, v in enumerate(half):
                out[ch, q, d.index(v)] = lc[i]
                out[ch, q, d.index((-v[0], -v[1]))] = lc[i].mH
    return out, d


def _projected(spec, X, dev):
    """A_P, A_C of a state: the bare vertex, the channel itself and the gathers of the other channels' bond transforms."""
    F, n, L, Nq = spec.n_ff, spec.n_s, spec.Lq, spec.Nq
    n2 = n * n
    bonds = [tuple(int(x) for x in b) for b in spec.ff_R]
    at = {(b[0] % L, b[1] % L): i for i, b in enumerate(bonds)}
    qx, qy = torch.arange(Nq, device=dev) // L, torch.arange(Nq, device=dev) % L

    def phase(v):
        a = (qx * v[0] + qy * v[1]) % L
        return torch.polar(torch.ones(Nq, dtype=torch.float64, device=dev), 2 * math.pi * a.double() / L)

    seen = {}

    def bond(ch, v):   # X(R) = (1/Nq) sum_u e^{iu.R} X(u), indexed [i1][pair1][i2][pair2]
        k = (ch, v[0] % L, v[1] % L)
        if k not in seen:
            seen[k] = (phase(v) @ X[ch].reshape(Nq, -1) / Nq).reshape(F, n, n, F, n, n)
        return seen[k]

    def find(x, y):
        return at.get((x % L, y % L), -1)

    classes = sorted({((a[0] - b[0]) % L, (a[1] - b[1]) % L) for a in bonds for b in bonds})
    A = X.clone().reshape(2, Nq, F, n2, F, n2)
    for ch, V in enumerate(_pair_matrices(spec, dev)):
        A[ch][:, 0, :, 0, :] += V
    for r, R in enumerate(bonds):
        for p, P in enumerate(bonds):
            for out in (0, 1):
                ps, ms = [], []
                for c in classes:
                    i1, i2, j2 = find(R[0] + c[0], R[1] + c[1]), find(P[0] - c[0], P[1] - c[1]), find(-P[0] - c[0], -P[1] - c[1])
                    if i1 >= 0 and i2 >= 0:
                        ps.append(phase(c))
                        B = bond(1 - out, c)[i1, :, :, i2]
                        # P <- C: (s1 s3),(s4 s2) -> (s1 s2),(s4 s3);  C <- P: (s1 s2),(s4 s3) -> (s1 s3),(s4 s2)
                        ms.append(B.permute(0, 3, 2, 1))
                    if out == 0 and i1 >= 0 and j2 >= 0:
                        ps.append(-phase((P[0] + c[0], P[1] + c[1])))
                        B = bond(1, c)[i1, :, :, j2]                   # (s1 s4),(s3 s2) -> (s1 s2),(s4 s3)
                        ms.append(B.permute(0, 3, 1, 2))
                if out == 1:
                    for i2, W in enumerate(bonds):
                        i1 = find(R[0] - P[0] + W[0], R[1] - P[1] + W[1])
                        if i1 >= 0:
                            ps.append(-phase(W))
                            B = bond(1, (-P[0], -P[1]))[i1, :, :, i2]  # (s1 s4),(s3 s2) -> (s1 s3),(s4 s2)
                            ms.append(B.permute(0, 2, 1, 3))
                if ps:
                    m = torch.stack([b.reshape(-1) for b in ms])
                    A[out][:, r, :, p, :] += (torch.stack(ps, 1) @ m).reshape(Nq, n2, n2)
    return A.reshape(2, Nq, F * n2, F * n2)


def _exact_mlp(case, seed, dev):
    p, X, Y = _net(case, seed)
    dims = [20] + [case["width"]] * case["depth"] + [1600]
    p, h, Y = torch.from_numpy(p).to(dev), torch.from_numpy(X).to(dev).double(), torch.from_numpy(Y).to(dev).double()
    leaves, o = [], 0
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        W = p[o:o + a * b].to(torch.bfloat16).double().reshape(a, b).requires_grad_()   # the weights are BF16
        v = p[o + a * b:o + a * b + b].double().requires_grad_()
        o += a * b + b
        leaves += [W, v]
        h = h @ W + v
        if i < len(dims) - 2:
            h = torch.nn.functional.gelu(h)
    loss = ((h - Y) ** 2).mean()
    g = torch.autograd.grad(loss, leaves)
    return {"loss": float(loss), "grad": torch.cat([x.reshape(-1) for x in g])}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed, dev)
    if case["kind"] == "flow":   # hundreds of right-hand sides
        return None
    ns = {"hubbard": 2, "rashba": 2, "bilayer": 4, "t2g": 6}[case["family"]]
    Nq, Nk = case["Lq"] ** 2, (case["Lq"] * case["nc"]) ** 2
    if 2.0 * Nq * Nk * (21 + ns) * ns ** 4 * 8 > 4e12 or Nq * (case["n_ff"] * ns * ns) ** 3 > 2e10:
        return None
    spec = _spec(case, seed)
    A = _projected(spec, _state(case, spec, seed, dev), dev)
    Lc, d = _loops(spec, case["T"], case["shell"], dev)
    F, n2 = spec.n_ff, ns * ns
    idx = torch.tensor([[d.index((int(a[0] - b[0]), int(a[1] - b[1]))) for b in spec.ff_R] for a in spec.ff_R], device=dev)
    out = torch.empty_like(A)
    for ch in (0, 1):
        for q0 in range(0, Nq, 64):
            Lm = Lc[ch, q0:q0 + 64][:, idx].permute(0, 1, 3, 2, 4).reshape(-1, F * n2, F * n2)
            a = A[ch, q0:q0 + 64]
            out[ch, q0:q0 + 64] = (ch + 1) * (a @ Lm @ a)
    return out
