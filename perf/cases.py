"""The work that a user of this library has it do, as a list of cases to time.

A user builds a model (diabatic surfaces, bath, hierarchy depth), makes a `Propagator`, brings the ground
state to equilibrium, propagates and reads response functions, spectra and states.  The cases below do
that through the public entry points at the sizes of this repository's workloads: a 32 x 32 harmonic
model (one linear response; the batched 2D spectrum), a 96 x 128 photoisomerization model of depth 8,
the paper's 512 x 128 Morse model, a 256 x 256 three-state model of depth 10, a heterogeneous batch, and
the learned closure (propagation with it, one training gradient).  The arithmetic forms are the FP64 form
(the default), the mixed form (FP32 stages, FP64 zeroth tier) and the split-bf16 tensor-core form.

Results of the mixed forms are returned in single precision, which is what they carry: their traces come
from FP32 stages, so digits past the seventh are rounding.

`exact` restates the equations in 64 bits with torch (FFT along p, finite differences, classic RK4)
without this repository's code.
"""
import math

import numpy as np
import torch

from paper_1706_09590_gb300 import qhfpe

TRUNCATE, TERMINATOR, LEARNED = 0, 1, 2
HIDDEN, N_COEF, N_STATS = 256, 10, 67


# ---- the cases -----------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest calls: one propagation of the 32 x 32 model (16,384 cells), where a step is a few
        # microseconds of work and launches and dependent latency count; in the reference arithmetic
        dict(name="absorption 32x32 fp64", kind="response1", model="harmonic", nq=32, np=32, depth=3, eta=0.5,
             precision="fp64", steps=200),
        # and in the mixed form
        dict(name="absorption 32x32 mixed", kind="response1", model="harmonic", nq=32, np=32, depth=3, eta=0.5,
             precision="mixed", steps=200),
        # the batched 2D spectrum at full size: 64 t1 x 4 t2 x 2 pathways = 512 replicas, 512 t3 steps, and the
        # double Fourier transform of every waiting time
        dict(name="2D spectrum 32x32 mixed", kind="response3", model="harmonic", nq=32, np=32, depth=3, eta=0.5,
             precision="mixed", n_t1=64, stride=8, n_t2=4, t2_step=100, steps=512, n_omega=64),
        # the photoisomerization model at 96 x 128, depth 8, two Matsubara terms (8.1 M cells): steps from a
        # given state with the trace recorded, the state read back
        dict(name="steps 96x128 d8 mixed", kind="steps", model="photoiso", nq=96, np=128, depth=8, eta=1.0,
             precision="mixed", steps=24),
        dict(name="steps 96x128 d8 fp64", kind="steps", model="photoiso", nq=96, np=128, depth=8, eta=1.0,
             precision="fp64", steps=4),
        dict(name="steps 96x128 d8 bf16x3", kind="steps", model="photoiso", nq=96, np=128, depth=8, eta=1.0,
             precision="bf16x3", steps=12),
        # the largest: three states, 256 x 256, depth 10 (286 elements, 168.7 M cells, 1.35 GB in FP32)
        dict(name="steps 256x256 S3 mixed", kind="steps", model="three_state", nq=256, np=256, depth=10, eta=1.0,
             precision="mixed", steps=4),
        # the paper's own Morse model, underdamped bath (1.6 M cells, resident in L2)
        dict(name="absorption morse mixed", kind="response1", model="morse", nq=512, np=128, depth=5, eta=0.4,
             precision="mixed", steps=200),
        # equilibration of the ground state (always FP64, one surface, full hierarchy), which comes before every
        # response; a grid whose row count is no multiple of any tile
        dict(name="equilibrate 97x128 d8", kind="equilibrate", model="photoiso", nq=97, np=128, depth=8, eta=1.0,
             precision="mixed", steps=40),
        # a bath scan as one heterogeneous batch: eight models of different grids (odd row counts among them),
        # depths, closures and time steps
        dict(name="hetero batch np32 mixed", kind="batch", members=8, np=32, nq_lo=24, nq_hi=47, depth_lo=2, depth_hi=6,
             precision="mixed", steps=100),
        # the learned closure deployed: depth 4 on 96 x 128, FP64
        dict(name="learned closure 96x128", kind="response1", model="harmonic", nq=96, np=128, depth=4, eta=0.3,
             precision="fp64", closure="learned", steps=40),
        # one gradient of the closure network over all grid points of a bath (FP32 forward and backward)
        dict(name="closure gradient 96x128", kind="gradient", points=96 * 128, ridge=0.01),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _elements(depth, modes):
    return math.comb(depth + modes, modes)


def draw(rng):
    kind = rng.choice(["response1", "response1", "steps", "steps", "steps", "response3", "equilibrate", "batch",
                       "gradient"])
    if kind == "gradient":
        return dict(kind=kind, points=_log_int(rng, 700, 12288), ridge=rng.choice([0.0, 0.01]))
    if kind == "batch":
        lo = rng.randint(16, 33)
        return dict(kind=kind, members=rng.randint(2, 8), np=rng.choice([32, 64]), nq_lo=lo, nq_hi=lo + rng.randint(0, 14),
                    depth_lo=2, depth_hi=rng.randint(3, 6), precision=rng.choice(["mixed", "mixed", "fp64"]),
                    steps=rng.randint(17, 60))
    if kind == "response3":
        return dict(kind=kind, model="harmonic", nq=rng.randint(24, 48), np=rng.choice([32, 64]), depth=rng.randint(2, 4),
                    eta=round(rng.uniform(0.2, 1.0), 3), precision=rng.choice(["mixed", "mixed", "fp64"]),
                    n_t1=rng.randint(2, 10), stride=rng.randint(2, 8), n_t2=rng.randint(1, 3), t2_step=rng.randint(5, 30),
                    steps=rng.randint(20, 50), n_omega=rng.randint(16, 64))
    if kind == "equilibrate":
        m = rng.choice(["harmonic", "photoiso"])
        return dict(kind=kind, model=m, nq=rng.randint(31, 110), np=rng.choice([32, 64, 128]),
                    depth=rng.randint(2, 8), eta=round(rng.uniform(0.2, 1.0), 3), precision=rng.choice(["fp64", "mixed"]),
                    steps=rng.randint(8, 40))
    if kind == "response1":
        m = rng.choice(["harmonic", "harmonic", "photoiso", "morse"])
        c = dict(kind=kind, model=m, nq=_log_int(rng, 24, 100), np=rng.choice([32, 64, 128]), depth=rng.randint(2, 5),
                 eta=round(rng.uniform(0.2, 1.0), 3), precision=rng.choice(["fp64", "mixed"]), steps=rng.randint(17, 80))
        if m == "morse":
            c.update(nq=rng.randint(200, 512), np=128, precision="mixed")
        if m == "harmonic" and rng.random() < 0.3:
            c["closure"] = "learned"
        return c
    # steps: log-uniform over the state sizes
    three = rng.random() < 0.3
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64", "bf16x3"])
    if prec == "bf16x3":
        three = False
    if three:
        c = dict(kind=kind, model="three_state", nq=_log_int(rng, 33, 256), np=rng.choice([64, 128, 256]),
                 depth=rng.randint(3, 7), precision="mixed" if prec == "bf16x3" else prec)
    else:
        c = dict(kind=kind, model="photoiso", nq=_log_int(rng, 30, 130),
                 np=rng.choice([64, 128] if prec == "bf16x3" else [32, 64, 128, 256]), depth=rng.randint(2, 8), precision=prec)
    c["eta"] = round(rng.uniform(0.1, 1.0), 3)
    cells = _elements(c["depth"], 3) * (9 if three else 4) * c["nq"] * c["np"]
    budget = 3e7 if c["precision"] == "fp64" else 2e8  # cell-updates of one pass, at most
    c["steps"] = max(1, min(rng.randint(4, 40), int(budget / cells)))
    return c


# ---- models: surfaces, bath and grid of this repository's workloads ---------------------------------------
def _continued(f, lo, hi, h=1e-5):
    """f inside [lo, hi], its tangents outside (the potential kernel samples U beyond the box)."""
    flo, fhi = f(lo), f(hi)
    slo, shi = (f(lo + h) - f(lo - h)) / (2 * h), (f(hi + h) - f(hi - h)) / (2 * h)

    def g(q):
        out = f(np.clip(q, lo, hi))
        out = np.where(q < lo, flo + slo * (q - lo), out)
        return np.where(q > hi, fhi + shi * (q - hi), out)

    return g


def _model(c, seed):
    """The model dict that Propagator takes, and its potential table.  The seed moves the ground
    surface, the diabatic coupling and the energy gap by a few percent."""
    r = np.random.RandomState(seed % (1 << 32))
    a, b = 1.0 + 0.05 * r.uniform(-1, 1), 1.0 + 0.02 * r.uniform(-1, 1)
    kind = c["model"]
    well = lambda q: 5.0 * b * ((q / 4.0) ** 2 - 1.0) ** 2
    exc = lambda q: 0.5 * (q - 3.0) ** 2 + 0.01 * (q - 3.0) ** 4 - 0.31 * b
    m = dict(nq=c["nq"], np=c["np"], eta=c["eta"], depth=c["depth"], periodic_q=0, mu=np.array([[0.0, 1.0], [1.0, 0.0]]), S=2)
    if kind == "harmonic":
        m.update(q_min=-8.0, q_max=8.0, p_min=-8.0, p_max=8.0, gamma=1.0, beta=0.48, n_matsubara=0, high_temperature=1,
                 use_cdelta=0, closure=TERMINATOR, dt=0.01 if c["np"] <= 64 else 0.003)
        U = [[lambda q: 0.5 * b * q * q, lambda q: 0.5 * a + 0 * q],
             [lambda q: 0.5 * a + 0 * q, lambda q: 0.5 * (q - 1.5) ** 2 + 10.0 * b]]
    elif kind == "photoiso":
        m.update(q_min=-10.0, q_max=10.0, p_min=-16.0, p_max=16.0, gamma=1.0, beta=1.0, n_matsubara=2, high_temperature=0,
                 use_cdelta=1, closure=TRUNCATE, dt=1.6e-3 if c["np"] <= 128 else 8e-4)
        U = [[_continued(well, -10.0, 10.0), lambda q: 0.5 * a + 0 * q],
             [lambda q: 0.5 * a + 0 * q, _continued(exc, -10.0, 10.0)]]
    elif kind == "three_state":
        m.update(S=3, q_min=-10.0, q_max=10.0, p_min=-16.0, p_max=16.0, gamma=2.0, beta=0.5, n_matsubara=2,
                 high_temperature=0, use_cdelta=1, closure=TRUNCATE, dt=6.5e-4,
                 mu=np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 0.0], [1.0, 0.0, 0.0]]))
        v = lambda q: 0.5 * a + 0 * q
        U = [[_continued(well, -10.0, 10.0), v, v], [v, _continued(exc, -10.0, 10.0), v],
             [v, v, _continued(lambda q: exc(q - 1.0) + 2.0, -10.0, 10.0)]]
    else:  # the paper's Morse diabats with a Gaussian coupling
        a0, a1 = 1.0 / math.sqrt(1400.0), 0.8 / math.sqrt(1000.0)
        m.update(q_min=-20.0, q_max=80.0, p_min=-25.0, p_max=25.0, gamma=5.0, beta=0.48, n_matsubara=0, high_temperature=1,
                 use_cdelta=0, closure=TERMINATOR, dt=1e-3)
        v = lambda q: 6.0 * a * np.exp(-(q - 10.28) ** 2 / 8.0)
        U = [[lambda q: 700.0 * b * (1 - np.exp(-a0 * q)) ** 2, v],
             [v, lambda q: 500.0 * (1 - np.exp(-a1 * (q - 18.98))) ** 2 + 10.0 * b]]
    if c.get("closure") == "learned":
        m["closure"] = LEARNED
    if "dt" in c:
        m["dt"] = c["dt"]
    if "terminator" in c:
        m["closure"] = TERMINATOR if c["terminator"] else TRUNCATE
    dp = (m["p_max"] - m["p_min"]) / m["np"]
    q = m["q_min"] + np.arange(m["nq"]) * ((m["q_max"] - m["q_min"]) / m["nq"])
    s = (np.arange(m["np"] + 1) - m["np"] / 2) * (math.pi / (m["np"] * dp))
    x = q[:, None] + s[None, :]
    return m, np.array([[U[j][k](x) for k in range(m["S"])] for j in range(m["S"])])


def _hierarchy(m):
    """All index vectors up to the depth: by tier, then lexicographic with the first mode's largest first."""
    def tier(modes, left):
        if modes == 1:
            return [(left,)]
        return [(v,) + t for v in range(left, -1, -1) for t in tier(modes - 1, left - v)]
    return [n for t in range(m["depth"] + 1) for n in tier(m["n_matsubara"] + 1, t)]


def _axes(m, device="cuda"):
    q = m["q_min"] + torch.arange(m["nq"], dtype=torch.float64, device=device) * ((m["q_max"] - m["q_min"]) / m["nq"])
    p = m["p_min"] + torch.arange(m["np"], dtype=torch.float64, device=device) * ((m["p_max"] - m["p_min"]) / m["np"])
    return q, p


def _state(m, seed, dtype):
    """A seeded state [elem][S][S][nq][np] on the GPU: in every block a wave packet (a Gaussian with a phase
    along q and p), smaller with each tier of the hierarchy."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    S, tiers = m["S"], torch.tensor([float(sum(n)) for n in _hierarchy(m)], device="cuda", dtype=torch.float64)
    E = len(tiers)
    u = torch.rand((6, E, S, S, 1, 1), generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    q, p = _axes(m)
    mid, half = 0.5 * (m["q_min"] + m["q_max"]), (m["q_max"] - m["q_min"]) / 20.0
    x = (q[:, None] - mid) / half
    amp = (0.6 ** tiers).reshape(E, 1, 1, 1, 1) * (1.0 + 0.3 * u[0]) * torch.exp(1j * math.pi * u[1])
    pw = (m["p_max"] - m["p_min"]) / 16.0
    w = torch.empty((E, S, S, m["nq"], m["np"]), dtype=dtype, device="cuda")
    for e in range(E):  # an element at a time: the largest state is 1.3 GB
        f = torch.exp(-0.25 * (x - 1.5 * u[2, e]) ** 2 - 0.5 * ((p[None, :] - pw * u[3, e]) / pw) ** 2)
        w[e] = (amp[e] * f * torch.exp(1j * (0.8 * u[4, e] * x + 0.7 * u[5, e] * p[None, :] / pw))).to(dtype)
    return w


def _equilibrium(m, T, seed):
    """A ground-state distribution [elem][S][S][nq][np] (numpy): the Boltzmann distribution of the first
    surface, and in the tiers above its p-derivative-shaped corrections with seeded sizes."""
    r = np.random.RandomState(seed % (1 << 32))
    q, p = (x.numpy() for x in _axes(m, "cpu"))
    U = T[0, 0, :, m["np"] // 2]
    f = np.exp(-m["beta"] * (0.5 * p[None, :] ** 2 + (U - U.min())[:, None]))
    f /= f.sum() * (q[1] - q[0]) * (p[1] - p[0])
    H = _hierarchy(m)
    W = np.zeros((len(H), m["S"], m["S"], m["nq"], m["np"]), dtype=np.complex128)
    for e, n in enumerate(H):
        W[e, 0, 0] = f if e == 0 else f * (0.1 * r.uniform(-1, 1) * p[None, :]) * 0.3 ** sum(n)
    return W


def _network(seed):
    """The closure network's flat weights (three hidden layers of 256, Glorot-uniform; a small output layer)."""
    r = np.random.RandomState(seed % (1 << 32))
    parts = []
    for out, inp in ((HIDDEN, 3), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (N_COEF, HIDDEN)):
        lim = math.sqrt(6.0 / (out + inp)) * (0.02 if out == N_COEF else 1.0)
        parts += [r.uniform(-lim, lim, out * inp), 0.01 * r.uniform(-1, 1, out)]
    return np.concatenate(parts).astype(np.float32)


def _layers(w):
    """[(matrix, bias)] of the flat weights."""
    out, at = [], 0
    for o, i in ((HIDDEN, 3), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (N_COEF, HIDDEN)):
        out.append((w[at:at + o * i].reshape(o, i), w[at + o * i:at + o * i + o]))
        at += o * i + o
    return out


def _training(c, seed):
    """Network inputs (q/8, p/8, ln eta) and regression statistics of `points` grid points: the normal matrix
    (upper triangle), right-hand side, squared sum and count of twelve complex samples of ten regressors."""
    r = np.random.RandomState(seed % (1 << 32))
    n = c["points"]
    X = np.stack([r.uniform(-1, 1, n), r.uniform(-1, 1, n), np.full(n, math.log(0.3))], axis=1)
    phi, y = r.standard_normal((n, 12, 10)), r.standard_normal((n, 12))
    G, h = np.einsum("nsa,nsb->nab", phi, phi), np.einsum("nsa,ns->na", phi, y)
    a, b = np.triu_indices(10)
    return X, np.concatenate([G[:, a, b], h, (y * y).sum(1)[:, None], np.full((n, 1), 12.0)], axis=1)


def _members(c, seed):
    """The members of a heterogeneous batch, spread over the case's row counts and depths."""
    out = []
    for k in range(c["members"]):
        f = k / max(1, c["members"] - 1)
        out.append(dict(model="harmonic", nq=int(round(c["nq_lo"] + f * (c["nq_hi"] - c["nq_lo"]))), np=c["np"],
                        depth=c["depth_lo"] + (k * 3) % (c["depth_hi"] - c["depth_lo"] + 1), eta=0.2 + 0.2 * k,
                        terminator=k % 2 == 0, dt=(0.008 + 0.0005 * k) * 32 / c["np"]))
    return [(mc, seed * 16 + k) for k, mc in enumerate(out)]


# ---- one pass ----------------------------------------------------------------------------------------------
def _dtype(c):
    return torch.complex128 if c["precision"] == "fp64" else torch.complex64


def prepare(case, seed):
    c = case
    if c["kind"] == "gradient":
        X, stats = _training(c, seed)
        return dict(c=c, w=_network(seed), X=X, stats=stats)
    if c["kind"] == "batch":
        made = [_model(mc, s) for mc, s in _members(c, seed)]
        props = [qhfpe.Propagator(m, T, precision=c["precision"]) for m, T in made]
        states = [_state(m, seed * 16 + k, _dtype(c)) for k, (m, T) in enumerate(made)]
        torch.cuda.synchronize()
        return dict(c=c, props=props, batch=qhfpe.Batch(props), W=states, out=[torch.empty_like(w) for w in states])
    m, T = _model(c, seed)
    P = qhfpe.Propagator(m, T, precision=c["precision"])
    s = dict(c=c, P=P, m=m)
    if c.get("closure") == "learned":
        P.closure_load(_network(seed))
    if c["kind"] in ("response1", "response3"):
        P.set_equilibrium(_equilibrium(m, T, seed))
    if c["kind"] == "steps":
        s["W"] = _state(m, seed, _dtype(c))
    if c["kind"] in ("steps", "equilibrate"):
        s["out"] = torch.empty(P.shape, dtype=_dtype(c), device="cuda")
    if c["kind"] == "response3":
        s["t2"] = [b * c["t2_step"] for b in range(c["n_t2"])]
        s["omega"] = _omega(c)
    torch.cuda.synchronize()
    return s


def _omega(c):
    return np.linspace(4.0, 16.0, c["n_omega"])


def _carried(c, x):
    """A host result in the precision that the arithmetic form carries."""
    return x if c["precision"] == "fp64" else x.astype(np.complex64 if np.iscomplexobj(x) else np.float32)


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "gradient":
        loss, grad = qhfpe.closure_loss_grad(s["w"], s["X"], s["stats"], ridge=c["ridge"])
        return [np.float32(loss), grad]
    if c["kind"] == "batch":
        for P, W in zip(s["props"], s["W"]):
            P.set_state(W)
        tr = s["batch"].step(c["steps"], record_trace=True)
        return [[_carried(c, t) for t in tr], [P.get_state(0, out=o) for P, o in zip(s["props"], s["out"])]]
    P = s["P"]
    if c["kind"] == "response1":
        return _carried(c, P.linear_response(c["steps"]))
    if c["kind"] == "response3":
        R = P.third_order_response(c["n_t1"], c["stride"], s["t2"], c["steps"], split_pathways=True)
        dt = s["m"]["dt"]
        maps = [P.spectrum_2d(R[0, b] + R[1, b], c["stride"] * dt, dt, s["omega"], s["omega"])[:2] for b in range(c["n_t2"])]
        return [_carried(c, R), [[_carried(c, x) for x in m] for m in maps]]
    if c["kind"] == "equilibrate":
        res = P.equilibrate(c["steps"])
        return [np.float32(res), P.get_state(0, out=s["out"])]
    P.set_state(s["W"])
    tr = P.step(c["steps"], record_trace=True)
    return [_carried(c, tr), P.get_state(0, out=s["out"])]


# ---- bytes and operations that a pass cannot do without ------------------------------------------------------
L2_BYTES = 126e6


def _propagation(m, S, replicas, steps, real_bytes):
    """RK4 of `replicas` states: four right-hand sides a step.  A state that does not fit in the cache is read
    and written in each (eleven passes a step: input, result, and the step's start for three of the four
    combinations); one that does is read and written once."""
    modes = m["n_matsubara"] + 1
    E = _elements(m["depth"], modes)
    cells = float(E) * S * S * m["nq"] * m["np"] * replicas
    state = 2 * real_bytes * cells
    # two transforms along p (5 log2 N each), the S x S products, the six-point q difference, the tier
    # couplings (up and down neighbours, the p difference) and the update, for a complex value
    neighbours = 2.0 * modes * m["depth"] / (m["depth"] + modes)
    flops = 10 * math.log2(m["np"]) + 4 * (2 * S - 1) + 26 + 4 * neighbours + 14 + 4
    return dict(bytes=(11.0 * steps if 3 * state > L2_BYTES else 2.0) * state, flops=4.0 * steps * flops * cells)


def work(case):
    c = case
    if c["kind"] == "gradient":
        n = c["points"]
        macs = n * (3 * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN * N_COEF)
        # forward; weight gradients; input gradients of all layers but the first
        return dict(bytes=8.0 * n * (3 + N_STATS) + 8.0 * _network(0).size, flops=2.0 * (3 * macs - n * 3 * HIDDEN))
    rb = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "batch":
        parts = [_propagation(_model(mc, s)[0], 2, 1, c["steps"], rb) for mc, s in _members(c, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    m, _ = _model(c, 0)
    if c["kind"] == "equilibrate":
        return _propagation(m, 1, 1, c["steps"], 8)
    if c["kind"] == "response3":
        parts = [_propagation(m, 2, 2, c["stride"] * (c["n_t1"] - 1), rb),
                 _propagation(m, 2, 2 * c["n_t1"], c["t2_step"] * (c["n_t2"] - 1), rb),
                 _propagation(m, 2, 2 * c["n_t1"] * c["n_t2"], c["steps"], rb)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _propagation(m, m["S"], 1, c["steps"], rb)


# ---- the same in 64 bits, with torch --------------------------------------------------------------------------
class _Exact:
    """The equations of motion for states [..., elem, S, S, nq, np] in complex128."""

    def __init__(self, m, T, coef=None, device="cuda"):
        self.m, self.S = m, T.shape[0]
        self.q, self.p = _axes(m, device)
        self.dq, self.dp = (m["q_max"] - m["q_min"]) / m["nq"], (m["p_max"] - m["p_min"]) / m["np"]
        N = m["np"]
        T = torch.as_tensor(np.ascontiguousarray(T), device=device)
        k = torch.arange(N, device=device)
        k = torch.where(k < N // 2, k, k - N)  # the mode at each position of the transform
        self.UL, self.UR = T[..., k + N // 2].clone(), T[..., N // 2 - k].clone()
        edge = 0.5 * (T[..., 0] + T[..., N])
        self.UL[..., N // 2] = edge
        self.UR[..., N // 2] = edge
        self.coef = coef
        # bath
        eta, g, beta, K = m["eta"], m["gamma"], m["beta"], m["n_matsubara"]
        gam, r, cc, delta = [g], [eta], [eta / beta], 0.0
        if not m["high_temperature"]:
            cc = [0.5 * eta * g / math.tan(0.5 * beta * g)]
            for n in range(1, K + 1):
                nu = 2 * math.pi * n / beta
                gam.append(nu)
                r.append(0.0)
                cc.append(2 * eta * g * g / beta / (nu * nu - g * g))
            delta = eta / beta - sum(cc) if m["use_cdelta"] else 0.0
        self.gam, self.r, self.cc, self.delta = gam, r, cc, delta
        self.H = _hierarchy(m)
        self.index = {n: e for e, n in enumerate(self.H)}

    def d1(self, x):
        R = lambda s: torch.roll(x, s, -1)
        return (R(2) - 8 * R(1) + 8 * R(-1) - R(-2)) / (12 * self.dp)

    def d2(self, x):
        R = lambda s: torch.roll(x, s, -1)
        return (-R(2) + 16 * R(1) - 30 * x + 16 * R(-1) - R(-2)) / (12 * self.dp ** 2)

    def upwind(self, x):
        n = x.shape[-2]
        z = torch.nn.functional.pad(torch.view_as_real(x), (0, 0, 0, 0, 3, 3))
        z = torch.view_as_complex(z.contiguous())
        s = lambda d: z[..., 3 + d:3 + d + n, :]
        neg = 2 * s(3) - 15 * s(2) + 60 * s(1) - 20 * s(0) - 30 * s(-1) + 3 * s(-2)
        pos = -3 * s(2) + 30 * s(1) + 20 * s(0) - 60 * s(-1) + 15 * s(-2) - 2 * s(-3)
        return torch.where(self.p < 0, neg, pos) / (60 * self.dq)

    def element(self, W, e):
        """dW/dt of one element; W: [..., elem, S, S, nq, np]."""
        n, m, w = self.H[e], self.m, W[..., e, :, :, :, :]
        out = -self.p * self.upwind(w)
        rho = torch.fft.ifft(w)
        if self.S == 1:
            c = (self.UL[0, 0] - self.UR[0, 0]) * rho
        else:
            c = torch.einsum("jsim,...skim->...jkim", self.UL.to(rho.dtype), rho)
            c -= torch.einsum("...jsim,skim->...jkim", rho, self.UR.to(rho.dtype))
        out += torch.fft.fft(-1j * c)
        out -= sum(a * g for a, g in zip(n, self.gam)) * w
        if self.delta:
            out += self.delta * self.d2(w)
        G = torch.zeros_like(w)
        for k in range(len(n)):
            up = self.index.get(n[:k] + (n[k] + 1,) + n[k + 1:])
            if up is not None:
                G = G + W[..., up, :, :, :, :]
            if n[k]:
                x = W[..., self.index[n[:k] + (n[k] - 1,) + n[k + 1:]], :, :, :, :]
                G = G + n[k] * self.gam[k] * self.cc[k] * x
                if self.r[k]:
                    out += n[k] * self.gam[k] * self.r[k] * self.p * x
        if m["closure"] != TRUNCATE and sum(n) == m["depth"]:
            G = G + self.r[0] * self.p * w
            out += self.cc[0] * self.d2(w)
            if self.coef is not None:
                low = W[..., e - 1, :, :, :, :] if e else None
                for b in range(-2, 3):
                    G = G + self.coef[..., 2 + b] * torch.roll(w, -b, -1)
                    if low is not None:
                        G = G + self.coef[..., 7 + b] * torch.roll(low, -b, -1)
        return out + self.d1(G)

    def rhs(self, W):
        return torch.stack([self.element(W, e) for e in range(len(self.H))], dim=-5)

    def step(self, W, dt):
        v = W
        for k in (4, 3, 2, 1):
            v = W + (dt / k) * self.rhs(v)
        return v

    def dipole(self, W, side):
        mu = torch.as_tensor(self.m["mu"], device=W.device).to(W.dtype)
        left = torch.einsum("jl,...lkim->...jkim", mu, W) if side != "right" else 0
        right = torch.einsum("...jlim,lk->...jkim", W, mu) if side != "left" else 0
        return left - right if side == "both" else left + right

    def trace(self, W):
        mu = torch.as_tensor(self.m["mu"], device=W.device).to(W.dtype)
        return torch.einsum("kj,...jk->...", mu, W[..., 0, :, :, :, :].sum((-1, -2))) * (self.dq * self.dp)

    def propagate(self, W, steps, dt):
        tr = [self.trace(W)]
        for _ in range(steps):
            W = self.step(W, dt)
            tr.append(self.trace(W))
        return W, torch.stack(tr, -1)


def _bf16(x):
    return x.to(torch.bfloat16).to(torch.float64)


def _coefficients(m, w, device="cuda"):
    """The network at every grid point, with the bf16-rounded weights and activations it is served with."""
    q, p = _axes(m, device)
    h = torch.stack([(q / 8)[:, None].expand(-1, m["np"]), (p / 8)[None, :].expand(m["nq"], -1),
                     torch.full((m["nq"], m["np"]), math.log(m["eta"]), device=device, dtype=torch.float64)], -1).float()
    h = _bf16(h)
    for k, (A, b) in enumerate(_layers(w)):
        h = h @ _bf16(torch.as_tensor(A, device=device)).T + torch.as_tensor(b, device=device).double()
        if k < 3:
            h = _bf16(torch.tanh(h).float())
    return h


def exact(case, seed):
    c = case
    if c["kind"] == "gradient":
        X, stats = _training(c, seed)
        X, st = torch.as_tensor(X, device="cuda"), torch.as_tensor(stats, device="cuda")
        w = torch.as_tensor(_network(seed), device="cuda").double().requires_grad_(True)
        h = X.float().double()
        for k, (A, b) in enumerate(_layers(w)):
            h = h @ A.T + b
            h = torch.tanh(h) if k < 3 else h
        a, b = np.triu_indices(10)
        G = torch.zeros((len(X), 10, 10), dtype=torch.float64, device="cuda")
        G[:, a, b] = st[:, :55]
        G[:, b, a] = st[:, :55]
        ridge = c["ridge"] * torch.diagonal(G, dim1=1, dim2=2).sum(1) / 10.0
        loss = (torch.einsum("na,nab,nb->n", h, G, h) - 2 * (h * st[:, 55:65]).sum(1) + st[:, 65] + ridge * (h * h).sum(1)).sum()
        loss = loss / st[:, 66].sum()
        loss.backward()
        return [loss.detach(), w.grad]
    if c["kind"] == "batch":
        if sum(mc["depth"] for mc, _ in _members(c, seed)) * c["steps"] > 4000:
            return None
        tr, out = [], []
        for k, (mc, s) in enumerate(_members(c, seed)):
            m, T = _model(mc, s)
            W, t = _Exact(m, T).propagate(_state(m, seed * 16 + k, _dtype(c)).to(torch.complex128), c["steps"], m["dt"])
            tr.append(t[None])
            out.append(W)
        return [tr, out]
    m, T = _model(c, seed)
    coef = _coefficients(m, _network(seed)) if c.get("closure") == "learned" else None
    dt = m["dt"]
    if c["kind"] == "equilibrate":
        E = _Exact(m, T[:1, :1], coef)
        q, p = _axes(m)
        U = torch.as_tensor(T[0, 0, :, m["np"] // 2].copy(), device="cuda")
        f = torch.exp(-m["beta"] * (0.5 * p[None, :] ** 2 + U[:, None]))
        W = torch.zeros((len(E.H), 1, 1, m["nq"], m["np"]), dtype=torch.complex128, device="cuda")
        W[0, 0, 0] = f / (f.sum() * E.dq * E.dp)
        for _ in range(c["steps"]):
            W = E.step(W, dt)
        res = torch.linalg.vector_norm(E.rhs(W)) / torch.linalg.vector_norm(W)
        full = torch.zeros((len(E.H), m["S"], m["S"], m["nq"], m["np"]), dtype=torch.complex128, device="cuda")
        full[:, 0, 0] = W[:, 0, 0]
        return [res, full]
    E = _Exact(m, T, coef)
    if c["kind"] == "steps":
        W, tr = E.propagate(_state(m, seed, _dtype(c)).to(torch.complex128), c["steps"], dt)
        return [tr[None], W]
    W = torch.as_tensor(_equilibrium(m, T, seed), device="cuda")
    if c["kind"] == "response1":
        return 1j * E.propagate(E.dipole(W, "both"), c["steps"], dt)[1]
    cells = 2.0 * c["n_t1"] * c["n_t2"] * W.numel()
    if cells * c["steps"] > 1.5e9:
        return None  # the batched spectrum at full size takes minutes this way
    X, snaps = torch.stack([E.dipole(W, "left"), -E.dipole(W, "right")]), []
    for a in range(c["n_t1"]):
        for _ in range(c["stride"] if a else 0):
            X = E.step(X, dt)
        snaps.append(X)
    X, forks = E.dipole(torch.stack(snaps, 1), "both"), []
    for b in range(c["n_t2"]):
        for _ in range(c["t2_step"] if b else 0):
            X = E.step(X, dt)
        forks.append(X)
    R = -1j * E.propagate(E.dipole(torch.stack(forks, 1), "both"), c["steps"], dt)[1]  # [path][t2][t1][t3 + 1]
    om = torch.as_tensor(_omega(c), device="cuda")
    n1, n3, dt1 = c["n_t1"], c["steps"] + 1, c["stride"] * dt

    def weights(n, h):
        w = torch.full((n,), h, dtype=torch.float64, device="cuda")
        w[0] *= 0.5
        w[-1] *= 0.5
        return w

    t1, t3 = torch.arange(n1, device="cuda") * dt1, torch.arange(n3, device="cuda") * dt
    E3, E1 = torch.exp(1j * om[:, None] * t3) * weights(n3, dt), torch.exp(1j * om[:, None] * t1)
    maps = []
    for b in range(c["n_t2"]):
        G = E3 @ (R[0, b] + R[1, b]).T
        w1 = weights(n1, dt1).to(G.dtype)
        maps.append([(G @ (E1 * w1).T).imag, (G @ (E1.conj() * w1).T).imag])
    return [R, maps]
