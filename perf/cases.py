"""The work that users of the solver have it do, as cases with inputs made from a seed.

A case names a kind of problem, its sizes, the state's precision and the call: ``step`` or
``solve`` (time evolution, then the observables), or a gradient.  Every case goes through the
public Python entry points; times are in ns, angular frequencies in rad/ns.

``exact`` restates the method on dense 64-bit complex matrices with plain torch: the adjoint
Lindblad equation of every separable initial condition in the number basis, classical RK4, and
torch's own reverse mode for the gradients.
"""

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2203_05526_gb300 as bq
from paper_2203_05526_gb300.autograd import measured_probability

TWO_PI = 2.0 * math.pi
BASIS_MONOMIAL, BASIS_NUMBER = "monomial", "number"

# N: truncation of an oscillator (of a batch: the largest, 10..N); steps: RK4 steps of one call.
LISTED = [
    # One RK4 step of the smallest system and its observable: a program that watches one damped
    # oscillator step by step.  Latency and launches are all of it.
    dict(name="one_kerr_one_step", kind="kerr", instances=1, N=16, driven=False, thermal=False, dtype="f64", call="step", steps=1),
    # The driven oscillator at finite temperature in FP64, stepped from Python in chunks.
    dict(name="one_kerr_driven_f64", kind="kerr", instances=1, N=40, thermal=True, dtype="f64", call="step", steps=64),
    # The same oscillator in FP32 through the one-launch solve: a whole horizon at a time.
    dict(name="one_kerr_driven_solve", kind="kerr", instances=1, N=40, thermal=True, dtype="f32", call="solve", steps=2000),
    # The ragged 4096-instance batch through the one-launch solve: parameter scans.
    dict(name="batch_solve", kind="kerr", instances=4096, N=40, thermal=False, dtype="f32", call="solve", steps=200),
    # A batch whose state is larger than L2, stepped: the streaming end of the range.
    dict(name="large_batch_step", kind="kerr", instances=16384, N=40, thermal=False, dtype="f32", call="step", steps=64),
    # The batch in FP64: the spot checks that go with every FP32 scan.
    dict(name="batch_step_f64", kind="kerr", instances=1024, N=40, thermal=False, dtype="f64", call="step", steps=16),
    # The paper's own (secular) dissipator on the batch, stepped a few steps between read-outs.
    dict(name="secular_batch_step", kind="secular", instances=4096, N=40, thermal=False, dtype="f32", call="step", steps=20),
    # Two exchange-coupled modes in FP64, schedule tuned on the state before the run.
    dict(name="two_mode_step", kind="two_mode", N=12, method="mapped", dtype="f64", call="step", steps=100, tune=True),
    # The conventional number-basis method on three coupled modes (the paper's comparison).
    dict(name="network_direct", kind="network", modes=3, N=6, method="direct", layout="full", dtype="f64", call="step", steps=32),
    # The same network mapped, every initial condition of a_1 a_2 a_3 at once, R(xy) layout.
    dict(name="network_mapped", kind="network", modes=3, N=6, method="mapped", layout="diag", dtype="f64", call="step", steps=32),
    # The 131-parameter control gradient, schedule tuned on the gradient: one optimiser step.
    dict(name="control_grad", kind="control", instances=1, N=12, steps=320, segments=64, every=160, call="grad", tune=True),
    # Loss and gradient through torch.autograd with default schedules, small modes.
    dict(name="control_autograd", kind="control", instances=1, N=7, steps=96, segments=16, every=32, call="autograd", tune=False),
]


def listed():
    return [dict(c) for c in LISTED]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["kerr_one", "kerr_batch", "kerr_batch", "kerr_f64", "secular", "two_mode", "network", "control"])
    if kind == "kerr_one":
        return dict(kind="kerr", instances=1, N=rng.randint(8, 42), driven=rng.random() < 0.7, thermal=rng.random() < 0.5,
                    dtype=rng.choice(["f64", "f32"]), call=rng.choice(["step", "solve"]), steps=_log_int(rng, 1, 1000))
    if kind in ("kerr_batch", "secular"):
        n = _log_int(rng, 100, 12000)
        return dict(kind="kerr" if kind == "kerr_batch" else "secular", instances=n, N=rng.randint(14, 40),
                    thermal=kind == "kerr_batch" and rng.random() < 0.3, dtype="f32", call=rng.choice(["step", "solve"]),
                    steps=_log_int(rng, 1, 100))
    if kind == "kerr_f64":
        return dict(kind="kerr", instances=_log_int(rng, 20, 1500), N=rng.randint(12, 40), thermal=rng.random() < 0.3,
                    dtype="f64", call=rng.choice(["step", "solve"]), steps=_log_int(rng, 1, 20))
    if kind == "two_mode":
        return dict(kind="two_mode", N=rng.randint(5, 13), method=rng.choice(["mapped", "direct"]),
                    dtype=rng.choice(["f64", "f64", "f32"]), call="step", steps=_log_int(rng, 4, 150),
                    tune=rng.random() < 0.5)
    if kind == "network":
        modes = rng.choice([2, 3])
        method = rng.choice(["mapped", "direct"])
        return dict(kind="network", modes=modes, N=rng.randint(4, 7 if modes == 2 else 6), method=method,
                    layout=rng.choice(["diag", "off"]) if method == "mapped" else "full", dtype="f64", call="step",
                    steps=_log_int(rng, 4, 100))
    call = rng.choice(["grad", "autograd"])
    segments = rng.choice([4, 7, 16, 32])  # a whole number of steps each
    return dict(kind="control", instances=1 if call == "autograd" else rng.choice([1, 1, 3]), N=rng.randint(4, 10),
                steps=segments * max(1, _log_int(rng, 20, 200) // segments), segments=segments,
                every=rng.choice([16, 32, 50]), call=call, tune=False)


# ---- problem descriptions -----------------------------------------------------------------
# A problem is a namespace with the fields that the binding reads: modes, truncations,
# normal-ordered terms (a^dag)^u a^v, jump operators, envelopes and the measured operator.
# Truncations belong to the case, every physical parameter to the seed.

def _unit(n, j, p):
    return tuple(p if i == j else 0 for i in range(n))


def _term(coef, u, v, channel=-1, conj=False, param=-1):
    return SimpleNamespace(coef=complex(coef), u=u, v=v, channel=channel, conj=conj, param=param)


class _Channel:
    def __init__(self, kind, params):
        self.kind, self.params = kind, tuple(params)


def _problem(n, N, h, measured, T, dt, jumps=(), secular=(), channels=(), params=()):
    return SimpleNamespace(n_modes=n, N=N, h_terms=list(h), jumps=list(jumps), secular=list(secular), measured=measured,
                           channels=list(channels), params=list(params), rho0=None, reverse_time=True, T=T, dt=dt,
                           n_steps=int(round(T / dt)))


def _drive(n, j, ch):
    return [_term(1.0, _unit(n, j, 1), _unit(n, j, 0), ch, False), _term(1.0, _unit(n, j, 0), _unit(n, j, 1), ch, True)]


def _jump(rate, u, v):
    return SimpleNamespace(rate=rate, terms=((1.0 + 0j, u, v),))


def _truncations(case):
    """The truncation of every instance: the case's N for one, 10..N spread evenly for a batch."""
    if case["instances"] == 1:
        return [case["N"]]
    return [int(x) for x in np.random.RandomState(case["instances"]).randint(10, case["N"] + 1, case["instances"])]


def _kerr_problems(case, seed):
    """Damped Kerr oscillators with or without a Gaussian drive: detuning, anharmonicity,
    damping, drive peak and measured level |n><n| from the seed."""
    rng = np.random.RandomState(seed % (1 << 32))
    Ns = _truncations(case)
    top = max(Ns)
    dt = min(0.01, 2.4 / (TWO_PI * 0.125 * top * (top - 1) + 4.0 * math.sqrt(top)))
    horizon = 100.0  # t = horizon - tau: the run starts 10 ns after the pulse's centre
    out = []
    for N in Ns:
        delta = rng.uniform(-TWO_PI * 0.01, TWO_PI * 0.01)
        kerr = rng.uniform(-TWO_PI * 0.25, -TWO_PI * 0.15)
        gamma = 10.0 ** rng.uniform(-4.0, -3.0)
        peak = rng.uniform(0.1, 1.0) * TWO_PI * 0.05
        level = int(rng.randint(0, 3))
        a = (1,)
        h = [_term(delta, a, a), _term(kerr / 2.0, (2,), (2,))]
        channels, jumps, secular = [], [], []
        if case.get("driven", True):
            channels = [_Channel("gauss", (peak, 0.0, horizon - 10.0, 10.0))]
            h += _drive(1, 0, 0)
        if case["kind"] == "secular":
            secular = [SimpleNamespace(mode=0, kappa=gamma, nbar=())]
        else:
            n_th = 0.05 if case["thermal"] else 0.0
            jumps = [_jump(gamma * (1.0 + n_th), (0,), a)] + ([_jump(gamma * n_th, a, (0,))] if n_th else [])
        out.append(_problem(1, (N,), h, {((level,), (level,)): 1.0 + 0j}, horizon, dt, jumps, secular, channels))
    return out


def _two_modes(case, seed, control=False):
    """Two exchange-coupled Kerr modes; control: K_1, K_2, g as parameters and a complex
    piecewise-constant drive on mode 1."""
    out = []
    for b in range(case.get("instances", 1)):
        rng = np.random.RandomState((seed + 7919 * b) % (1 << 32))
        N = case["N"]
        kerr = -TWO_PI * 0.2 * (1.0 + 0.1 * rng.uniform(-1, 1, 2))
        g = TWO_PI * 0.005 * (1.0 + 0.2 * rng.uniform(-1, 1))
        delta = TWO_PI * 0.1 * (1.0 + 0.1 * rng.uniform(-1, 1))
        h = [_term(delta, (0, 1), (0, 1))]
        params = [float(kerr[0]), float(kerr[1]), float(g)] if control else []
        for j in range(2):
            h.append(_term(0.5 if control else kerr[j] / 2.0, _unit(2, j, 2), _unit(2, j, 2), param=j if control else -1))
        for u, v in (((1, 0), (0, 1)), ((0, 1), (1, 0))):
            h.append(_term(1.0 if control else g, u, v, param=2 if control else -1))
        jumps = [_jump(1e-4, (0, 0), _unit(2, j, 1)) for j in range(2)]
        channels, dt, T = [], 0.01, 100.0
        if control:
            dt = 0.008
            T = case["steps"] * dt
            amp = rng.normal(0.0, TWO_PI * 0.01, 2 * case["segments"])
            # every segment is met: the pulse is as long as the run
            channels = [_Channel("pwc", (0.0, T / case["segments"], *[float(x) for x in amp]))]
            h += _drive(2, 0, 0)
        out.append(_problem(2, (N, N), h, {((1, 0), (1, 0)): 1.0 + 0j}, T, dt, jumps, (), channels, params))
        if control:  # the second mode excited in part of the runs: the loss feels g as well as the drive
            out[-1].rho0 = {((0, 0), (0, 0)): 0.7 + 0j, ((0, 1), (0, 1)): 0.3 + 0j}
    return out


def _network(case, seed):
    """Coupled anharmonic oscillators in the lab frame (Eq. 301 with the values of Table I, each
    spread by a few per cent), mode 1 driven by a complex exponential, secular dissipator at zero
    temperature, A(0) = a_1 (x) ... (x) a_n."""
    n, N = case["modes"], case["N"]
    rng = np.random.RandomState(seed % (1 << 32))
    w, eta, J, om = (TWO_PI * x * (1.0 + 0.05 * rng.uniform(-1, 1)) for x in (3.5, 0.25, 0.01, 0.125))
    h = []
    for j in range(n):
        h += [_term(w, _unit(n, j, 1), _unit(n, j, 1)), _term(eta, _unit(n, j, 2), _unit(n, j, 2))]
        for k in range(j + 1, n):
            h += [_term(J, _unit(n, k, 1), _unit(n, j, 1)), _term(J, _unit(n, j, 1), _unit(n, k, 1))]
    z, a1 = _unit(n, 0, 0), _unit(n, 0, 1)
    h += [_term(1j * om, z, a1, 0, False), _term(-1j * om, a1, z, 0, True)]
    measured = {}
    for k in np.ndindex(*([N - 1] * n)):
        k = tuple(int(x) for x in k)
        measured[(k, tuple(x + 1 for x in k))] = complex(math.prod(math.sqrt(x + 1) for x in k))
    T = 10.0 * math.pi / w
    return [_problem(n, (N,) * n, h, measured, T, T / 2000, (), [SimpleNamespace(mode=j, kappa=2e-5, nbar=()) for j in range(n)],
                     [_Channel("cexp", (1.0, 0.0, w))])]


def _problems(case, seed):
    if case["kind"] in ("kerr", "secular"):
        return _kerr_problems(case, seed)
    if case["kind"] == "network":
        return _network(case, seed)
    return _two_modes(case, seed, control=case["kind"] == "control")


# ---- the calls ------------------------------------------------------------------------------
def _opts(case, p):
    return dict(method=case.get("method", "mapped"), dtype=case.get("dtype", "f64"), r_layout=case.get("layout", "full"),
                reverse_time=p.reverse_time, horizon=p.T, dt=p.dt)


def prepare(case, seed):
    probs = _problems(case, seed)
    p = probs[0]
    st = SimpleNamespace(case=case, dt=p.dt, steps=case["steps"])
    if case["call"] == "autograd":
        st.spec = p
        st.theta = torch.tensor(p.params, dtype=torch.float64, requires_grad=True)
        st.pwc = torch.tensor(p.channels[0].params[2:], dtype=torch.float64).reshape(-1, 2).requires_grad_()
        return st
    st.state = bq.State([bq.problem_from_spec(q) for q in probs], bq.map_opts(**_opts(case, p)))
    if case["call"] == "grad":
        if case["tune"]:
            st.state.autotune_grad(p.dt, trial_steps=16, checkpoint_every=8)
        return st
    if case.get("tune"):
        st.state.autotune(p.dt)
    st.host = torch.empty(st.state.state_bytes(), dtype=torch.uint8, pin_memory=True)
    return st


def run(st):
    """The state's arrays and Tr(rho0 A) of every problem after the call; or loss and gradient."""
    case = st.case
    if case["call"] == "autograd":
        st.theta.grad = st.pwc.grad = None
        loss = measured_probability(st.spec, st.theta, st.pwc, checkpoint_every=case["every"])
        loss.backward()
        return {"loss": loss.detach(), "theta": st.theta.grad, "pwc": st.pwc.grad}
    if case["call"] == "grad":
        loss, grad = st.state.grad(st.dt, st.steps, checkpoint_every=case["every"])
        return {"loss": loss, "grad": grad}
    getattr(st.state, case["call"])(st.dt, st.steps)
    st.state.store_state(st.host.data_ptr())
    trace = st.state.evaluate()  # waits for the stream, the copy before it included
    f32 = case["dtype"] == "f32"
    return {"state": st.host.view(torch.float32 if f32 else torch.float64),
            "trace": trace.astype(np.complex64) if f32 else trace}


# ---- the least work ---------------------------------------------------------------------------
def _sizes(case):
    """(grid points, stencil entries per point of R besides the diagonal) of all systems."""
    if case["kind"] in ("kerr", "secular"):
        return sum(N * N + 2 * N for N in _truncations(case)), 5
    n = 2 if case["kind"] != "network" else case["modes"]
    ng = case["N"] ** n
    if case.get("method") == "direct":
        return ng * ng, 2 * (n * (n - 1) + 2 if case["kind"] == "network" else 2) + n
    sep = case["kind"] == "network"
    systems = (case["N"] - 1) ** n if sep else case["instances"] if "instances" in case else 1
    r = {"full": ng * ng, "diag": ng, "off": 0}[case.get("layout", "full")]
    return systems * (r + 2 * ng), 2 * (n * (n - 1) + 2) + n if sep else (8 if case["kind"] == "control" else 4) + n


def work(case):
    """Bytes: the state read and written once.  Operations: a complex multiply-add (8) per
    stencil entry and point, the diagonal and the RK4 update, four stages a step; a gradient takes
    the forward stage, its transpose and the parameter sums."""
    points, entries = _sizes(case)
    size = 8 if case.get("dtype") == "f32" else 16
    passes = 3 if case["call"] in ("grad", "autograd") else 1
    return {"bytes": 2 * points * size, "flops": passes * 4 * case["steps"] * points * (8 * entries + 16)}


# ---- 64-bit restatement -------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _mono(u, v, N):
    """<k|(a^dag)^u a^v|l> for k, l < N."""
    m = np.zeros((N, N))
    for l in range(v, N):
        k = l - v + u
        if k < N:
            m[k, l] = math.sqrt(math.prod(range(l - v + 1, l + 1)) * math.prod(range(l - v + 1, k + 1)))
    return m


def _op(u, v, Ns):
    m = np.ones((1, 1))
    for j, N in enumerate(Ns):
        m = np.kron(m, _mono(u[j], v[j], N))
    return m


def _separation(p, k, l, om, et):
    """C of Eq. 304 for the initial condition x^k y^l."""
    return -0.5j * sum((om[j] - et[j]) * (k[j] + l[j]) + et[j] * (k[j] ** 2 + l[j] ** 2) for j in range(p.n_modes))


def _envelope(ch, t, t_mid, values=None):
    p = ch.params
    if ch.kind == "gauss":
        return complex(p[0], p[1]) * math.exp(-((t - p[2]) ** 2) / (2.0 * p[3] ** 2))
    if ch.kind == "cexp":
        return complex(p[0], p[1]) * complex(math.cos(p[2] * t), math.sin(p[2] * t))
    s = math.floor((t_mid - p[0]) / p[1])
    if not 0 <= s < (len(p) - 2) // 2:
        return 0.0
    return torch.complex(values[s, 0], values[s, 1]) if values is not None else complex(p[2 + 2 * s], p[3 + 2 * s])


class _Exact:
    """A batch of systems of equal layout on one padded grid: left operators X(t) = X0 + e X1 +
    conj(e) X2 by their non-zero diagonals, sandwich operators, G_x, G_y, R."""

    def __init__(self, probs, case, dev, theta=None, values=None):
        self.dev, self.case, self.theta, self.values = dev, case, theta, values
        self.direct = case.get("method") == "direct"
        self.layout = "full" if self.direct else case.get("layout", "full")
        self.p0 = probs[0]
        self.reach = max(math.prod(p.N) for p in probs)
        n = self.reach
        self.sys = []  # (problem, k, l)
        X, S, gx, gy, C, R, E = [], [], [], [], [], [], []
        for b, p in enumerate(probs):
            ng = math.prod(p.N)
            x = [np.zeros((n, n), complex) for _ in range(3)]
            self.dparam = []
            om, et = [0.0] * p.n_modes, [0.0] * p.n_modes
            for t in p.h_terms:
                m = 1j * t.coef * _op(t.u, t.v, p.N)
                if t.param >= 0:
                    self.dparam.append((t.param, torch.tensor(m, device=dev)))
                else:
                    x[0 if t.channel < 0 else 2 if t.conj else 1][:ng, :ng] += m
                one = [j for j in range(p.n_modes) if t.u[j] or t.v[j]]
                if t.channel < 0 and len(one) == 1:
                    c = t.coef.real * (theta[t.param] if theta is not None and t.param >= 0 else
                                       p.params[t.param] if t.param >= 0 else 1.0)
                    if t.u[one[0]] == t.v[one[0]] == 1:
                        om[one[0]] = om[one[0]] + c
                    if t.u[one[0]] == t.v[one[0]] == 2:
                        et[one[0]] = et[one[0]] + c
            s = []
            for jp in p.jumps:
                _, u, v = jp.terms[0]
                L = _op(u, v, p.N)
                # L^dag L as a normal-ordered polynomial: m for a, m + 1 for a^dag
                j = next(i for i in range(p.n_modes) if u[i] or v[i])
                k = np.unravel_index(np.arange(ng), p.N)[j].astype(float)
                x[0][np.arange(ng), np.arange(ng)] += -0.5 * jp.rate * (k if v[j] else k + 1.0)
                pad = np.zeros((n, n))
                pad[:ng, :ng] = math.sqrt(jp.rate) * L
                s.append((pad, None))
            for sd in p.secular:
                k = np.unravel_index(np.arange(ng), p.N)[sd.mode].astype(float)
                x[0][np.arange(ng), np.arange(ng)] += -0.5 * sd.kappa * k
                pad = np.zeros((n, n))
                pad[:ng, :ng] = math.sqrt(sd.kappa) * _op((0,) * p.n_modes, _unit(p.n_modes, sd.mode, 1), p.N)
                idx = np.full(n, -1.0)
                idx[:ng] = k
                s.append((pad, idx))
            ics = [None] if self.direct else sorted(p.measured)
            for ic in ics:
                self.sys.append((b, ic))
                X.append(x)
                S.append(s)
                a, c, r = np.zeros(n, complex), np.zeros(n, complex), None
                if self.direct:
                    r = np.zeros((n, n), complex)
                    for (k, l), v in p.measured.items():
                        r[np.ravel_multi_index(k, p.N), np.ravel_multi_index(l, p.N)] += v
                    C.append(0.0)
                else:
                    a[np.ravel_multi_index(ic[0], p.N)] = math.sqrt(math.prod(math.factorial(q) for q in ic[0]))
                    c[np.ravel_multi_index(ic[1], p.N)] = math.sqrt(math.prod(math.factorial(q) for q in ic[1]))
                    C.append(_separation(p, ic[0], ic[1], om, et))
                gx.append(a)
                gy.append(c)
                R.append(r)
        T = lambda v: torch.tensor(np.array(v), dtype=torch.complex128, device=dev)  # noqa: E731
        B = len(self.sys)
        same = all(x is X[0] for x in X)
        self.X = [self._diagonals(T([x[q] for x in (X[:1] if same else X)])) for q in range(3)]
        self.S = []
        for q in range(len(S[0])):
            Ld = T([s[q][0] for s in (S[:1] if same else S)]).conj().transpose(1, 2)
            mask = None
            if S[0][q][1] is not None:
                k = torch.tensor(np.array([s[q][1] for s in (S[:1] if same else S)]), device=dev)
                mask = (k[:, :, None] == k[:, None, :]).to(torch.complex128) if self.layout == "full" else True
            self.S.append((self._diagonals(Ld), mask))
        self.gx, self.gy = (None, None) if self.direct else (T(gx), T(gy))
        self.C = torch.stack([torch.as_tensor(c, dtype=torch.complex128, device=dev) for c in C])[:, None]
        self.R = T(R) if self.direct else (torch.zeros((B, n, n) if self.layout == "full" else (B, n), dtype=torch.complex128,
                                                       device=dev) if self.layout != "off" else None)
        self.chan = [p.channels[0] if p.channels else None for p in probs]
        self.one = all(c is None or c.params == self.chan[0].params for c in self.chan)

    @staticmethod
    def _diagonals(M):
        out = []
        n = M.shape[-1]
        for d in range(-n + 1, n):
            v = torch.diagonal(M, d, 1, 2)
            if torch.any(v != 0):
                out.append((d, v))
        return out

    @staticmethod
    def _left(diags, u, scale=None):
        """sum of the diagonals' products with u along dimension 1."""
        out = 0
        n = u.shape[1]
        for d, v in diags:
            w = v if scale is None else scale * v
            if u.dim() == 3:
                w = w[:, :, None]
            lo, hi = max(0, -d), n - max(0, d)
            out = out + torch.nn.functional.pad(w * u[:, lo + d:hi + d], ([0, 0] if u.dim() == 3 else []) + [lo, n - hi])
        return out if torch.is_tensor(out) else torch.zeros_like(u)

    def _apply(self, u, e):
        out = self._left(self.X[0], u)
        if e is not None:
            out = out + self._left(self.X[1], u, e) + self._left(self.X[2], u, e.conj())
        for q, m in self.dparam:
            th = self.theta[q] if self.theta is not None else self.p0.params[q]
            out = out + th * (m @ u if u.dim() == 3 else u @ m.T)
        return out

    def rhs(self, s, t, t_mid):
        gx, gy, R = s
        e = None
        if self.chan[0] is not None:
            v = [_envelope(c, t, t_mid, self.values) for c in (self.chan[:1] if self.one else self.chan)]
            e = (torch.stack([x if torch.is_tensor(x) else torch.tensor(x, dtype=torch.complex128, device=self.dev) for x in v])
                 .to(self.dev).to(torch.complex128)[:, None])
            if not self.one:
                e = e[[b for b, _ in self.sys]]
        dx = dy = None
        if gx is not None:
            dx = self._apply(gx, e) + self.C * gx
            dy = self._apply(gy.conj(), e).conj() - self.C * gy
        if R is None:
            return dx, dy, None
        if R.dim() == 2:  # R(xy): the k = l entries; no off-diagonal operator couples them
            dg = sum((v for d, v in self.X[0] if d == 0), torch.zeros((), dtype=torch.complex128, device=self.dev))
            dR = 2.0 * dg.real * R
            for Ld, _ in self.S:
                d, v = Ld[0]
                sh = lambda u: torch.nn.functional.pad(u[:, :d], [-d, 0])  # noqa: E731
                w = torch.nn.functional.pad(v, [-d, 0])
                dR = dR + w * w * (sh(R) + sh(gx) * sh(gy))
            return dx, dy, dR
        dR = self._apply(R, e) + self._apply(R.transpose(1, 2).conj(), e).transpose(1, 2).conj()
        src = R if gx is None else R + gx[:, :, None] * gy[:, None, :]
        for Ld, mask in self.S:
            v = self._left(Ld, self._left(Ld, src).transpose(1, 2).conj()).transpose(1, 2).conj()
            dR = dR + (v if mask is None else mask * v)
        return dx, dy, dR

    def steps(self, dt, n):
        y = (self.gx, self.gy, self.R)
        T = self.p0.T
        add = lambda a, s, k: tuple(None if u is None else u + s * v for u, v in zip(a, k))  # noqa: E731
        for i in range(n):
            tau = i * dt
            mid = T - (tau + 0.5 * dt)
            k1 = self.rhs(y, T - tau, mid)
            k2 = self.rhs(add(y, dt / 2, k1), T - (tau + 0.5 * dt), mid)
            k3 = self.rhs(add(y, dt / 2, k2), T - (tau + 0.5 * dt), mid)
            k4 = self.rhs(add(y, dt, k3), T - (tau + dt), mid)
            y = add(add(add(add(y, dt / 6, k1), dt / 3, k2), dt / 3, k3), dt / 6, k4)
        return y


def _factors(Ns, basis):
    if basis == BASIS_NUMBER:
        return np.ones(math.prod(Ns))
    k = np.unravel_index(np.arange(math.prod(Ns)), Ns)
    return np.prod([np.sqrt(np.array([float(math.factorial(int(q))) for q in kk])) for kk in k], axis=0)


def _exact_state(case, seed, dev):
    """State arrays [G_x | G_y | R] per system, each padded to four elements, and the traces."""
    probs = _problems(case, seed)
    basis = BASIS_MONOMIAL if case.get("method", "mapped") == "mapped" and case["dtype"] == "f64" else BASIS_NUMBER
    pieces, trace = [], np.zeros(len(probs), complex)
    chunk = len(probs) if len(probs) <= 2048 else 2048
    pad = lambda v: np.concatenate([v, np.zeros(-len(v) % 4, complex)])  # noqa: E731
    for b0 in range(0, len(probs), chunk):
        part = probs[b0:b0 + chunk]
        E = _Exact(part, case, dev)
        gx, gy, R = (None if v is None else v.cpu().numpy() for v in E.steps(part[0].dt, case["steps"]))
        for i, (b, ic) in enumerate(E.sys):
            p = part[b]
            ng, f = math.prod(p.N), _factors(p.N, basis)
            if gx is not None:
                pieces += [pad(gx[i, :ng] / f), pad(gy[i, :ng] / f)]
            if R is not None:
                pieces.append(pad(R[i, :ng] / f ** 2) if R.ndim == 2 else pad((R[i, :ng, :ng] / np.outer(f, f)).reshape(-1)))
            if ic is None:
                trace[b0 + b] += R[i, 0, 0]
            else:
                w = p.measured[ic] / math.sqrt(math.prod(math.factorial(q) for k in ic for q in k))
                trace[b0 + b] += w * (gx[i, 0] * gy[i, 0] + (0.0 if R is None else R[i].reshape(-1)[0]))
    v = np.concatenate(pieces)
    v = np.concatenate([v, np.zeros(max(0, 16 - len(v)), complex)])
    return {"state": torch.from_numpy(v.view(np.float64)), "trace": trace}


def _exact_grad(case, seed, dev):
    losses, grads = [], []
    for p in _problems(case, seed):
        theta = torch.tensor(p.params, dtype=torch.float64, device=dev, requires_grad=True)
        pwc = torch.tensor(p.channels[0].params[2:], dtype=torch.float64, device=dev).reshape(-1, 2).requires_grad_()
        E = _Exact([p], case, dev, theta, pwc)
        gx, gy, R = E.steps(p.dt, case["steps"])
        loss = sum(r.real * (gx[0, k] * gy[0, k] + R[0, k, k]).real
                   for k, r in ((np.ravel_multi_index(kl[0], p.N), r) for kl, r in p.rho0.items()))
        loss.backward()
        losses.append(loss.detach().cpu())
        grads.append((theta.grad.cpu(), pwc.grad.cpu()))
    if case["call"] == "autograd":
        return {"loss": losses[0], "theta": grads[0][0], "pwc": grads[0][1]}
    return {"loss": torch.stack(losses), "grad": torch.cat([torch.cat([a, b.reshape(-1)]) for a, b in grads])}


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] in ("grad", "autograd"):
        return _exact_grad(case, seed, dev)
    with torch.no_grad():
        return _exact_state(case, seed, dev)
