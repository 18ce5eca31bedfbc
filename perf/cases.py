"""The work that users have this framework do, as measurable cases.

A case is one call pattern of the public Python binding (``GPEPS``, ``KickedIsingZ``) on one
batch of lattices.  ``kind`` says which:

  evolve  a fresh evolution: ``reset``, ``step(steps, theta)``, ``expect_z``
  step    one Trotter step of a state in hand (a resumed checkpoint): ``load_state``,
          ``step(1, theta)``, ``expect_z``
  layer   the step's building block: ``load_state``, ``kick``, ``zz_layer(0)``, ``expect_z``
  weight  Weight-N observables by Clifford back-evolution: ``weight_z(theta, steps)``
  grad    d(sum_i w_i <Z_i>)/dtheta_i through the autograd function
  bp      one Trotter step followed by a belief-propagation regauge, and ``expect_z``

``lattice`` names the instances ("127", "433", "1121": the processors; "RxW": rows x width of the
heavy-hex rule; "cell": the 10-site unit cell of the infinite lattice), joined by "+", "*k"
repeating one.  ``schedule``, ``tensor``, ``floor32`` and ``floor_rel`` are the handle's settings
(absent: its defaults).

The states in hand are synthetic, made from the seed by torch alone: Schmidt spectra
lambda_k ~ exp(-a sqrt k) with a in [0.7, 1.05] per bond (which fits the spectra of the kicked
Ising evolution at theta = 0.7, D = 32 from step 10, a = 1.03, to steps 25 - 50, a = 0.73) and
complex Gaussian Gammas brought near the canonical form that the simple update keeps.

Outputs are gauge invariant: the mean-field <Z_i> and their means, the Schmidt spectra lambda
(decreasing per bond, as the update stores them) and gradients.  The Gammas themselves are
defined up to a phase per bond index (and a rotation of degenerate ones), so no two programs
agree on them, and they enter through <Z_i>, which reads every one of their elements.  An
evolution from |0...0> leaves bonds of incomplete rank, whose zero Schmidt values are rounding,
so it returns <Z> only.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2309_15642_gb300.gpeps import GPEPS, KickedIsingZ
from workloads.heavyhex import LATTICES, heavy_hex, heavy_hex_cell, heavy_hex_cell_colour

MIX = "127+433+1121"


def listed():
    return [
        # the smallest run of the repository: plain complex128 at D = 4, where latency counts
        dict(name="eagle_d4", kind="evolve", lattice="127", D=4, dtype="c128", steps=5),
        # the sweep of kick angles of a figure, all angles in one batch, mixed precision
        dict(name="sweep16_d16", kind="evolve", lattice="127*16", D=16, dtype="mixed", steps=8, schedule=6),
        # a new user's run: the 127-qubit processor, mixed precision, the handle's default settings
        dict(name="eagle_d32_default", kind="evolve", lattice="127", D=32, dtype="mixed", steps=8),
        # the headline batch (three processors) in its tuned setting, one steady-state step
        dict(name="mix_d32", kind="step", lattice=MIX, D=32, dtype="mixed", schedule=6, tensor=True, floor32=1e-7,
             floor_rel=7e-8),
        # the same step in plain complex128, the reference arm of the headline number
        dict(name="mix_d32_c128", kind="step", lattice=MIX, D=32, dtype="c128", schedule=4),
        # the infinite lattice: 16 angles on the unit cell, complex128, default settings
        dict(name="cell16_d32_c128", kind="evolve", lattice="cell*16", D=32, dtype="c128", steps=5),
        # the large run: 1121 qubits at D = 64, mixed precision with tensor-core passes
        dict(name="condor_d64", kind="step", lattice="1121", D=64, dtype="mixed", schedule=4, tensor=True,
             floor_rel=3e-8),
        # the 127-qubit processor at D = 64 in complex128
        dict(name="eagle_d64_c128", kind="step", lattice="127", D=64, dtype="c128", schedule=4),
        # the largest bond dimension: one colour class of the 127-qubit lattice at D = 128
        dict(name="eagle_d128_layer", kind="layer", lattice="127", D=128, dtype="c128"),
        # training per-qubit angles: forward and backward, checkpoints every 5 steps
        dict(name="grad_d16", kind="grad", lattice="127", D=16, dtype="c128", steps=10, ckpt=5),
        # belief-propagation regauging after a Trotter step, mixed precision with tensor cores
        dict(name="bp_d32", kind="bp", lattice="127", D=32, dtype="mixed", schedule=4, tensor=True),
        # Weight-N observables (forward steps, then Clifford back-evolution) in complex128
        dict(name="weight_d16", kind="weight", lattice="127", D=16, dtype="c128", steps=5),
    ]


def draw(rng):
    while True:
        kind = rng.choices(["evolve", "step", "layer", "weight", "grad", "bp"], [3, 5, 1, 1, 1, 1])[0]
        lattice = "%dx%d" % (rng.choice([3, 5, 7, 9, 13]), rng.choice([7, 11, 15, 19, 27]))
        if rng.random() < 0.25:
            lattice = "cell*%d" % rng.randint(2, 24)
        top = {"grad": 16, "weight": 32, "evolve": 40, "bp": 32}.get(kind, 64)
        some = [4, 8, 16, 32, 64] if rng.random() < 0.4 else range(3, 65)
        D = min(some, key=lambda d, at=rng.uniform(math.log(3), math.log(64)): abs(math.log(d) - at))
        case = dict(kind=kind, lattice=lattice, D=D, dtype="c128" if kind == "grad" else rng.choice(["c128", "mixed"]))
        if kind in ("evolve", "weight"):
            case["steps"] = rng.randint(2, 6)
        if kind == "grad":
            case.update(steps=rng.randint(3, 8), ckpt=rng.randint(2, 5))
        if kind != "grad" and rng.random() < 0.6:
            case["schedule"] = rng.choice([1, 4])
        if case["dtype"] == "mixed" and D in (32, 64) and rng.random() < 0.5:
            case["tensor"] = True
        # complex128 runs at 0.2 of the mixed path's rate: bound the cost below the largest listed cases
        if D <= top and work(case)["flops"] <= (4e10 if case["dtype"] == "c128" else 2e11):
            return case


# ------------------------------------------------------------------ graphs
def _graphs(case):
    out, colours = [], []
    for part in case["lattice"].split("+"):
        name, _, times = part.partition("*")
        for _ in range(int(times or 1)):
            if name == "cell":
                out.append(heavy_hex_cell())
                colours.append(heavy_hex_cell_colour())
            else:
                out.append(heavy_hex(*(LATTICES[int(name)] if "x" not in name else map(int, name.split("x")))))
                colours.append(None)
    return out, colours


def _legs(graphs):
    """Per site over all instances: its (neighbour site, edge) in leg order; and every edge's two sites."""
    legs, ends = [], []
    for n, edges in graphs:
        s0, at = len(legs), [[] for _ in range(n)]
        for a, b in np.asarray(edges).tolist():
            at[a].append((s0 + b, len(ends)))
            at[b].append((s0 + a, len(ends)))
            ends.append((s0 + a, s0 + b))
        legs += [sorted(x) for x in at]
    return legs, ends


def _colours(graphs, given):
    """Greedy first-fit over edges sorted by (smaller, larger) label, unless given."""
    out = []
    for (n, edges), col in zip(graphs, given):
        e = [(min(a, b), max(a, b)) for a, b in np.asarray(edges).tolist()]
        c, used = [0] * len(e), [set() for _ in range(n)]
        for i in sorted(range(len(e)), key=lambda i: e[i]):
            if col is None:
                a, b = e[i]
                c[i] = next(k for k in range(9) if k not in used[a] | used[b])
                used[a].add(c[i])
                used[b].add(c[i])
            else:
                c[i] = int(col[i])
        out += c
    return out


# ------------------------------------------------------------------ inputs
def _angles(case, graphs, seed):
    """Kick angles: one per instance (clear of the Clifford point pi/2, where every Schmidt value
    ties), or one per qubit for the gradient."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "grad":
        return rng.uniform(0.5, 0.9, sum(n for n, _ in graphs))
    return rng.uniform(0.3, 1.1, len(graphs))


def _weights(graphs, seed):
    return np.random.default_rng([seed, 1]).uniform(0.5, 1.5, sum(n for n, _ in graphs))


def _state(case, graphs, seed):
    """Synthetic state in hand on the GPU: lambda (edges, D) in float64 and one Gamma per site."""
    D, cdt = case["D"], torch.complex128 if case["dtype"] == "c128" else torch.complex64
    legs, ends = _legs(graphs)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = 0.7 + 0.35 * torch.rand(len(ends), 1, generator=gen, device="cuda", dtype=torch.float64)
    lam = torch.exp(-a * torch.sqrt(torch.arange(D, device="cuda", dtype=torch.float64)))
    lam = lam / torch.linalg.vector_norm(lam, dim=1, keepdim=True)
    gamma = [None] * len(legs)
    for deg in (0, 1, 2, 3):
        sites = [i for i, x in enumerate(legs) if len(x) == deg]
        per = max(1, (1 << 26) // (2 * D ** deg))  # a bounded batch of sites at a time
        for at in range(0, len(sites), per):
            part = sites[at:at + per]
            t = torch.randn([len(part), 2] + [D] * deg, generator=gen, device="cuda", dtype=cdt)
            ws = [lam[[legs[i][q][1] for i in part]].to(t.real.dtype) for q in range(deg)]
            for q in range(deg):  # whiten leg q in the environment of the others
                A = t
                for p in range(deg):
                    if p != q:
                        A = A * ws[p].reshape([len(part), 1] + [D if r == p else 1 for r in range(deg)])
                A = A.movedim(q + 2, 1).reshape(len(part), D, -1)
                g = A @ A.mH
                g = g + 1e-3 * torch.eye(D, device="cuda") * g.diagonal(dim1=1, dim2=2).real.mean(1)[:, None, None]
                L = torch.linalg.cholesky(g)
                m = t.movedim(q + 2, 1)
                m = torch.linalg.solve_triangular(L, m.reshape(len(part), D, -1), upper=False).reshape(m.shape)
                t = m.movedim(1, q + 2)
            for k, i in enumerate(part):
                gamma[i] = t[k].contiguous()
    return lam, gamma


def prepare(case, seed):
    graphs, colours = _graphs(case)
    g = GPEPS(graphs, case["D"], case["dtype"], colours=colours)
    if case.get("schedule"):
        g.set_schedule(case["schedule"])
    if case.get("tensor"):
        g.set_tensor_cores(True)
    if "floor32" in case or "floor_rel" in case:
        g.set_jacobi(floor_rel=case.get("floor_rel"), floor32=case.get("floor32", 2e-7))
    state = dict(case=case, g=g, theta=torch.as_tensor(_angles(case, graphs, seed)).cuda())
    if case["kind"] in ("step", "layer", "bp"):
        lam, gamma = _state(case, graphs, seed)
        site = edge = 0
        for k, (n, edges) in enumerate(graphs):
            for v in range(n):
                g.site_tensor(k, v)[0].copy_(gamma[site + v])
            for e in range(len(edges)):
                g.lambda_tensor(k, e).copy_(lam[edge + e])
            site, edge = site + n, edge + len(edges)
        torch.cuda.synchronize()
        state["saved"] = g.state.clone()
        state["lam"] = g.state[:g.total_edges * g.D * 8].view(torch.float64).view(g.total_edges, g.D)
    elif case["kind"] == "grad":
        state["theta"].requires_grad_(True)
        state["w"] = torch.as_tensor(_weights(graphs, seed)).cuda()
    return state


def run(state):
    case, g, theta = state["case"], state["g"], state["theta"]
    kind = case["kind"]
    if kind == "evolve":
        g.reset()
        mean = g.step(case["steps"], theta)
        return [g.expect_z()[0], mean]
    if kind == "weight":
        return [g.weight_z(theta, case["steps"])]
    if kind == "grad":
        z = KickedIsingZ.apply(theta, g, case["steps"], case["ckpt"])
        (dtheta,) = torch.autograd.grad((z * state["w"]).sum(), theta)
        return [z.detach(), dtheta]
    g.load_state(state["saved"])
    if kind == "layer":
        g.kick(theta)
        g.zz_layer(0)
    else:
        g.step(1, theta)
        if kind == "bp":
            g.bp_regauge()
    z, mean = g.expect_z()
    return [z, mean, state["lam"]]


# ------------------------------------------------------------------ work
def _bonds(case):
    """(degree of the larger end, of the smaller end) of every bond that a pass's Trotter step updates."""
    graphs, given = _graphs(case)
    legs, ends = _legs(graphs)
    col = _colours(graphs, given) if case["kind"] == "layer" else [0] * len(ends)
    return legs, [sorted((len(legs[a]), len(legs[b])), reverse=True) for (a, b), c in zip(ends, col) if c == 0]


def work(case):
    """Per bond update, in complex multiply-adds (8 flops): the Gram (a Hermitian one) and the
    update of the larger end, R = D^(deg-1) rows; the core of the smaller end; a QR-based SVD of
    the n x 2D core with its right vectors (12 n^3 real-formula flops, x 4 for complex).  Bytes:
    each tensor of the state in and out once a step."""
    D, elt = case["D"], 16 if case["dtype"] == "c128" else 8
    legs, bonds = _bonds(case)
    flops = 0.0
    for da, db in bonds:
        R, n = D ** (da - 1), 2 * D ** (db - 1)
        flops += 8.0 * (R * D * D + 2 * R * D * D + 2 * D * n * D) + 48.0 * n ** 3
    state = sum(2.0 * D ** len(x) * elt for x in legs)
    times = case.get("steps", 1) * {"weight": 2, "grad": 3}.get(case["kind"], 1)
    if case["kind"] == "bp":  # one message per leg: the leg products and the Hermitian Gram, 8 iterations
        flops += 8 * sum(len(x) * 8.0 * (2 * (len(x) - 1) * D ** (len(x) + 1) + D ** (len(x) + 1)) for x in legs)
    return {"bytes": 2 * state * times, "flops": flops * times}


# ------------------------------------------------------------------ 64-bit values
def _pinv(lam):
    return torch.where(lam > 1e-13 * lam.max(), 1 / lam, torch.zeros_like(lam))


def _weighted(T, x, lam, skip, f):
    for p, (_, e) in enumerate(x):
        if p != skip:
            T = T * f(lam[e]).reshape([1] + [-1 if r == p else 1 for r in range(len(x))])
    return T


def _update(gamma, lam, legs, ends, e, D, phase):
    """Textbook simple update of edge e: absorb, QR, gate, SVD, truncate, renormalise, strip."""
    mats = []
    for i, j in (ends[e], ends[e][::-1]):
        p = [n for n, _ in legs[i]].index(j)
        A = _weighted(gamma[i], legs[i], lam, p, lambda v: v).movedim((0, p + 1), (-2, -1))
        Q, R = torch.linalg.qr(A.reshape(-1, 2 * D))
        mats.append((i, p, A.shape, Q, R.reshape(-1, 2, D)))
    (i, pi, si, Qi, Ri), (j, pj, sj, Qj, Rj) = mats
    th = torch.einsum("ask,btk->asbt", Ri * lam[e], Rj) * phase[None, :, None, :]
    U, S, Vh = torch.linalg.svd(th.reshape(2 * len(Ri), 2 * len(Rj)), full_matrices=False)
    keep = min(D, len(S))
    new = torch.zeros(D, dtype=torch.float64)
    new[:keep] = S[:keep] / torch.linalg.vector_norm(S[:keep])
    for site, p, shape, Q, W in ((i, pi, si, Qi, U[:, :keep]), (j, pj, sj, Qj, Vh[:keep].T)):
        T = torch.zeros(len(Q), 2, D, dtype=torch.complex128)
        T[:, :, :keep] = torch.einsum("ma,ask->msk", Q, W.reshape(-1, 2, keep))
        T = T.reshape(shape).movedim((-2, -1), (0, p + 1))
        gamma[site] = _weighted(T, legs[site], lam, p, _pinv)
    return e, new


def _kick(gamma, theta):
    for i, th in enumerate(theta):
        c, s = math.cos(th / 2), math.sin(th / 2)
        g0, g1 = gamma[i][0], gamma[i][1]
        gamma[i] = torch.stack([c * g0 - 1j * s * g1, c * g1 - 1j * s * g0])


def _layer(pool, gamma, lam, legs, ends, col, c, D, sign=1.0):
    phase = torch.exp(1j * sign * math.pi / 4 * torch.tensor([[1.0, -1.0], [-1.0, 1.0]], dtype=torch.complex128))
    todo = [e for e, k in enumerate(col) if k == c]
    for e, new in pool.map(lambda e: _update(gamma, lam, legs, ends, e, D, phase), todo):
        lam[e] = new


def _readout(gamma, lam, legs):
    z = []
    for i, x in enumerate(legs):
        p = _weighted(gamma[i], x, lam, -1, lambda v: v).reshape(2, -1).abs().square().sum(1)
        z.append(float((p[0] - p[1]) / (p[0] + p[1])))
    return np.array(z)


def _bp(pool, gamma, lam, legs, ends, D):
    """Belief propagation on the norm network to its fixed point, then the BP gauge of every edge."""
    back = {}
    for i, x in enumerate(legs):
        for p, (_, e) in enumerate(x):
            back[i, e] = p

    def send(msg, i, p):
        A = gamma[i]
        for q, (k, e) in enumerate(legs[i]):
            if q != p:
                env = lam[e][:, None] * msg[k, back[k, e]] * lam[e]
                A = torch.movedim(torch.tensordot(A, env, dims=([q + 1], [0])), -1, q + 1)
        A = A.movedim(p + 1, 0).reshape(D, -1)
        B = gamma[i].movedim(p + 1, 0).reshape(D, -1)
        m = A @ B.mH
        m = (m + m.mH) / 2
        on = (lam[legs[i][p][1]] > 1e-13 * lam[legs[i][p][1]].max()).to(m.dtype)
        m = m * on[:, None] * on
        return m / m.diagonal().sum().real

    keys = [(i, p) for i, x in enumerate(legs) for p in range(len(x))]
    msg = {k: torch.eye(D, dtype=torch.complex128) / D for k in keys}
    for _ in range(200):
        new = dict(zip(keys, pool.map(lambda k: send(msg, *k), keys)))
        far = max(float((new[k] - msg[k]).abs().max()) for k in keys)
        msg = new
        if far < 1e-13:
            break

    def root(m):
        w, v = torch.linalg.eigh(m.conj())
        on = w > 1e-13 * w.max()
        r = torch.where(on, w.clamp_min(0).sqrt(), 0)
        inv = torch.where(on, 1 / w.clamp_min(1e-300).sqrt(), 0)
        return (v * r) @ v.mH, (v * inv) @ v.mH

    def gauge(e):
        i, j = ends[e]
        (Ri, Pi), (Rj, Pj) = root(msg[i, back[i, e]]), root(msg[j, back[j, e]])
        U, S, Vh = torch.linalg.svd((Ri * lam[e]) @ Rj.T)
        on = (S > 1e-13 * S[0]).to(U.dtype)
        return S / torch.linalg.vector_norm(S), (Pi @ U) * on, (Pj @ Vh.T) * on

    for e, (s, gi, gj) in enumerate(list(pool.map(gauge, range(len(ends))))):
        lam[e] = s
        for i, m in zip(ends[e], (gi, gj)):
            p = back[i, e]
            gamma[i] = torch.movedim(torch.tensordot(gamma[i], m, dims=([p + 1], [0])), -1, p + 1)


def exact(case, seed):
    """The same quantities by the textbook simple update (QR and SVD of LAPACK) in 64 bits."""
    graphs, given = _graphs(case)
    kind, D = case["kind"], case["D"]
    times = case.get("steps", 1) * (2 if kind == "weight" else 1)
    if work(case)["flops"] > 6e11 or len(_bonds(case)[1]) * times > 25000 or (kind == "bp" and D > 32):
        return None  # more than about 20 seconds on the host
    legs, ends = _legs(graphs)
    col, theta = _colours(graphs, given), _angles(case, graphs, seed)
    if kind != "grad":
        theta = np.repeat(theta, [n for n, _ in graphs])
    if kind in ("step", "layer", "bp"):
        lam, gamma = _state(case, graphs, seed)
        lam, gamma = lam.cpu(), [t.cpu().to(torch.complex128) for t in gamma]
    else:
        lam = torch.zeros(len(ends), D, dtype=torch.float64)
        lam[:, 0] = 1
        gamma = [torch.zeros([2] + [D] * len(x), dtype=torch.complex128) for x in legs]
        for t in gamma:
            t[(0,) * t.dim()] = 1
    split = np.cumsum([n for n, _ in graphs])[:-1]
    threads = torch.get_num_threads()
    torch.set_num_threads(1)
    means = []
    with ThreadPoolExecutor(16) as pool:
        for _ in range(case.get("steps", 1)):
            _kick(gamma, theta)
            for c in range(1 if kind == "layer" else max(col) + 1):
                _layer(pool, gamma, lam, legs, ends, col, c, D)
            if kind == "evolve":
                means.append([float(x.mean()) for x in np.split(_readout(gamma, lam, legs), split)])
        if kind == "weight":
            for _ in range(case["steps"]):
                for c in range(max(col), -1, -1):
                    _layer(pool, gamma, lam, legs, ends, col, c, D, -1.0)
                _kick(gamma, -np.full(len(legs), math.pi / 2))
        if kind == "bp":
            _bp(pool, gamma, lam, legs, ends, D)
    torch.set_num_threads(threads)
    z = _readout(gamma, lam, legs)
    if kind == "evolve":
        return [z, np.array(means)]
    if kind == "weight":
        return [z]
    if kind == "grad":
        return [z, None]
    mean = np.array([x.mean() for x in np.split(z, split)])
    return [z, mean, lam.numpy()]
