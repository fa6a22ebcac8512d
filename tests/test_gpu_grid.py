"""The grid-resident kernels of the tiled path (bq_tune resident = 1) against the tiled kernels
(resident = 0) and the oracle: one to four modes, every residual layout, Hermitian and general
states, both precisions, gradients, and the forms they must leave to the tiled kernels."""

import dataclasses
import itertools

import numpy as np
import pytest

from oracle import grad as ograd
from oracle import mapping
from workloads import configs
from workloads.spec import Channel, HTerm, Jump, SecularDamping

from parity import compare_mapped_systems, gpu_state

pytestmark = pytest.mark.gpu
# two kernels' roundings over a few steps of O(1) data, as in the schedule tests: 1e-12 / 1e-6
TOL = {"f64": 1e-12, "f32": 1e-6}


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2203_05526_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _raw(st, dtype):
    import torch
    host = torch.empty(st.state_bytes(), dtype=torch.uint8, pin_memory=True)
    st.store_state(host.data_ptr())
    torch.cuda.synchronize()
    return host.numpy().view(np.float64 if dtype == "f64" else np.float32).astype(np.float64)


def _driven(N=5, drive="gauss", n_th=0.1, steps=11, secular=False, measured=None):
    """Two exchange-coupled, driven, damped Kerr modes."""
    p = configs.two_mode(N=N, T=steps * 0.005, dt=0.005)
    T = p.T
    p.channels = [{"gauss": Channel("gauss", (0.4, 0.1, 0.4 * T, 0.3 * T)), "cexp": Channel("cexp", (0.3, -0.1, 2.0)),
                   "const": Channel("const", (0.2, 0.1)),
                   "pwc": Channel("pwc", (0.0, T / 3, 0.3, 0.1, -0.2, 0.2, 0.1, -0.1))}[drive]]
    p.h_terms = p.h_terms + configs.gauss_drive_terms(2, 0, 0) + [HTerm(0.3, (1, 1), (1, 1))]  # and a cross-Kerr shift
    if secular:
        p.jumps = []
        p.secular = [SecularDamping(j, 0.05, (0.1,) * (N - 1) if n_th else ()) for j in range(2)]
    else:
        p.jumps = configs.damping_jumps(2, 0, 0.05, n_th) + configs.damping_jumps(2, 1, 0.03, n_th)
    if measured is not None:
        p.measured = measured
    return p


GENERAL = {((1, 0), (0, 1)): 0.7 + 0.2j, ((0, 0), (1, 0)): 0.5j, ((1, 1), (1, 1)): 1.0}


def _both(ps, dtype, steps, **kw):
    a, b = gpu_state(ps, dtype=dtype, **kw), gpu_state(ps, dtype=dtype, **kw)
    assert a.get_tune()["resident"] == 1 and a.get_tune()["stage_path"] == "tiled"
    b.set_tune(resident=0)
    dt = (ps if isinstance(ps, list) else [ps])[0].dt
    for st in (a, b):
        st.step(dt, steps - 2)
        st.step(dt, 2)
    return a, b


def _agree(a, b, dtype):
    x, y = _raw(a, dtype), _raw(b, dtype)
    assert np.all(np.isfinite(x))
    assert np.max(np.abs(x - y)) <= TOL[dtype] * np.max(np.abs(y))
    ea, eb = a.evaluate(), b.evaluate()
    assert np.max(np.abs(ea - eb)) <= TOL[dtype] * max(1.0, np.max(np.abs(eb)))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("measured", [None, GENERAL])
@pytest.mark.parametrize("form", [dict(), dict(drive="cexp"), dict(drive="pwc", n_th=0.0), dict(drive="const"),
                                  dict(secular=True), dict(secular=True, n_th=0.0), dict(N=2), dict(N=3), dict(N=6)])
def test_every_form_matches_the_tiled_kernels(dtype, measured, form):
    p = _driven(measured=measured, **form)
    a, b = _both(p, dtype, 11)
    _agree(a, b, dtype)
    if form == dict():
        compare_mapped_systems(a, mapping.rk4_mapped(p), 1e-10 if dtype == "f64" else 1e-5)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("kw", [dict(method="direct"), dict(r_layout="off"), dict(r_layout="diag")])
@pytest.mark.parametrize("modes", [1, 2, 3])
def test_layouts_and_modes(dtype, kw, modes):
    if modes == 1 and kw.get("r_layout") != "diag":
        pytest.skip("other single-mode states do not take the tiled path")
    p = configs.table_one_network(modes, 4, steps=4000)
    p = dataclasses.replace(p, T=12 * p.dt)
    a, b = _both(p, dtype, 12, **kw)
    _agree(a, b, dtype)


def test_four_modes_and_uneven_truncations():
    p = configs.table_one_network(4, 3, steps=4000)
    p = dataclasses.replace(p, T=6 * p.dt, measured={((1, 0, 1, 0), (0, 1, 1, 0)): 1.0 + 0.3j, ((1, 1, 0, 0), (1, 1, 0, 0)): 0.5})
    a, b = _both(p, "f64", 6)
    _agree(a, b, "f64")
    q = _driven()
    q.N = (7, 4)
    a, b = _both(q, "f64", 11)
    _agree(a, b, "f64")
    a, b = _both([_driven(N=5), _driven(N=3, n_th=0.0), _driven(N=4, measured=GENERAL)], "f64", 11)  # several problems
    _agree(a, b, "f64")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_loaded_states_and_switches(dtype):
    import torch
    p = _driven()
    a, b = _both(p, dtype, 9)
    snap = torch.from_numpy(_raw(a, dtype)).to(torch.float64 if dtype == "f64" else torch.float32)
    noise = torch.randn(snap.shape, generator=torch.Generator().manual_seed(5), dtype=torch.float64)
    n_g = p.N[0] * p.N[1]
    pad = (n_g + 3) & ~3
    keep = torch.zeros_like(snap)
    for off, n in ((0, n_g), (pad, n_g), (2 * pad, n_g * n_g)):  # the padding stays zero
        keep[2 * off:2 * (off + n)] = 1
    host = ((snap + 1e-2 * noise.to(snap.dtype)) * keep).contiguous().pin_memory()  # not Hermitian
    for st in (a, b):
        st.load_state(host.data_ptr())
        st.step(p.dt, 3)
    _agree(a, b, dtype)
    a.set_tune(resident=0)
    a.step(p.dt, 1)
    a.set_tune(resident=1)
    a.step(p.dt, 2)
    b.step(p.dt, 3)
    _agree(a, b, dtype)


def _control(N, B=1, n_seg=3, steps_per_seg=6, measured=None):
    ps = []
    for b in range(B):
        p = configs.two_mode_control(n_seg=n_seg, T=n_seg * steps_per_seg * 0.01, steps_per_seg=steps_per_seg, N=N, seed=5526 + b)
        p.jumps = configs.damping_jumps(2, 0, 0.05, 0.1) + configs.damping_jumps(2, 1, 0.03, 0.0)
        p.rho0 = {((0, 0), (0, 0)): 0.6, ((1, 0), (1, 0)): 0.3, ((0, 1), (1, 0)): 0.1j, ((1, 0), (0, 1)): -0.1j}
        if measured:
            p.measured = measured
        ps.append(p)
    return ps


@pytest.mark.parametrize("measured", [None, {((1, 0), (1, 0)): 1.0, ((1, 0), (0, 1)): 0.7 + 0.2j, ((0, 1), (1, 0)): 0.7 - 0.2j}])
@pytest.mark.parametrize("N,B,every", [(2, 1, 18), (4, 1, 7), (5, 3, 5), (7, 1, 1)])
def test_gradients_match_the_tiled_kernels_and_the_oracle(measured, N, B, every):
    ps = _control(N, B, measured=measured)
    a, b = gpu_state(ps), gpu_state(ps)
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    la, ga = a.grad(ps[0].dt, ps[0].n_steps, every)
    lb, gb = b.grad(ps[0].dt, ps[0].n_steps, every)
    assert np.max(np.abs(la - lb)) <= 1e-13 * max(1.0, np.max(np.abs(lb)))
    assert np.max(np.abs(ga - gb)) <= 1e-12 * np.max(np.abs(gb))
    if N == 4:
        loss, gt, gp = ograd.loss_and_grad(ps[0], checkpoint_every=every)
        ref = np.concatenate([gt, gp[0].reshape(-1)])
        assert abs(la[0] - loss) <= 1e-12 * max(1.0, abs(loss))
        assert np.max(np.abs(ga - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("kw", [dict(r_layout="diag"), dict(r_layout="off"), dict(method="direct")])
@pytest.mark.parametrize("secular", [False, True])
def test_gradients_of_other_layouts(kw, secular):
    p = _control(4)[0]
    if secular:
        p.jumps = []
        p.secular = [SecularDamping(j, 0.05, (0.1,) * 3) for j in range(2)]
    a, b = gpu_state(p, **kw), gpu_state(p, **kw)
    b.set_tune(resident=0)
    la, ga = a.grad(p.dt, p.n_steps, 5)
    lb, gb = b.grad(p.dt, p.n_steps, 5)
    assert abs(la[0] - lb[0]) <= 1e-13 * max(1.0, abs(lb[0]))
    assert np.max(np.abs(ga - gb)) <= 1e-12 * np.max(np.abs(gb))


def test_other_forms_keep_the_tiled_kernels():
    def one(f):
        p = _driven(N=3)
        f(p)
        st = gpu_state(p)
        st.set_tune(resident=1)
        return st.get_tune()["resident"]

    z, a = (0, 0), (1, 0)
    assert one(lambda p: None) == 1
    # a time-dependent diagonal term, a jump operator of two monomials
    assert one(lambda p: p.h_terms.extend([HTerm(0.2, a, a, channel=0), HTerm(0.2, a, a, channel=0, conj=True)])) == 0
    assert one(lambda p: p.jumps.append(Jump(0.1, ((1.0 + 0j, z, a), (0.5 + 0j, z, z))))) == 0


def test_independent_systems_drift_apart_without_losing_slots():
    """125 systems that no exchange couples, many blocks of steps and several calls: CTAs run ahead of
    one another as far as the slots' reuse lets them."""
    p = configs.table_one_network(3, 6, steps=4000)
    a, b = gpu_state(p, dtype="f64", r_layout="diag"), gpu_state(p, dtype="f64", r_layout="diag")
    b.set_tune(resident=0)
    for n in (61, 1, 2, 96):
        a.step(p.dt, n)
        b.step(p.dt, n)
    _agree(a, b, "f64")


@pytest.mark.parametrize("instances,N", [(1, 19), (1, 20), (1, 42), (2, 8), (31, 41), (128, 9), (129, 9)])
def test_few_single_mode_systems(instances, N):
    """FP64 single-mode states on both sides of the rule that sends few systems to the grid kernels."""
    ps = [configs.kerr_driven(N=max(4, N - i % 3), dt=0.002, T=0.05, n_th=0.1 if i % 2 else 0.0) for i in range(instances)]
    a, b = gpu_state(ps, dtype="f64"), gpu_state(ps, dtype="f64")
    b.set_tune(resident=0)
    for n in (1, 13):
        a.step(ps[0].dt, n)
        b.step(ps[0].dt, n)
    a.solve(ps[0].dt, 5)
    b.step(ps[0].dt, 5)
    _agree(a, b, "f64")


@pytest.mark.parametrize("N", [4, 14])
@pytest.mark.parametrize("every", [9, 10, 11, 12, 16, 17, 25])
def test_gradient_segments_of_every_remainder(N, every):
    """Segments of n steps with every n mod 8 that starts the backward sweep in a batch's lowest four
    steps (and 8 and 16 beside them), the pulse changing its value at every step: the parameter sums are
    reduced at each change.  Blocks of four steps (N = 4) and of two (N = 14)."""
    p = configs.two_mode_control(n_seg=25, T=25 * 0.005, steps_per_seg=1, N=N)
    p.rho0 = {((0, 0), (0, 0)): 0.7, ((1, 0), (0, 1)): 0.1j, ((0, 1), (1, 0)): -0.1j, ((1, 0), (1, 0)): 0.3}
    a, b = gpu_state(p), gpu_state(p)
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    la, ga = a.grad(p.dt, p.n_steps, every)
    lb, gb = b.grad(p.dt, p.n_steps, every)
    assert p.n_steps == 25
    assert abs(la[0] - lb[0]) <= 1e-13 * max(1.0, abs(lb[0]))
    assert np.max(np.abs(ga - gb)) <= 1e-12 * np.max(np.abs(gb))
    if N == 4:
        loss, gt, gp = ograd.loss_and_grad(p, checkpoint_every=every)
        ref = np.concatenate([gt, gp[0].reshape(-1)])
        assert np.max(np.abs(ga - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("modes", [1, 2])
def test_gradients_at_a_parameter_of_zero(modes):
    """theta = 0: the coefficients of theta's terms are 0, their derivatives are not (they differ between
    terms, which a comparison of coefficients alone does not see).  Two modes at N = 3, where
    (a_2^dag)^2 and a_1^dag a_2 shift the flat index alike; one mode with a drive and a detuning."""
    if modes == 2:
        p = _driven(3, drive="pwc")
        p.rho0 = {((0, 0), (0, 0)): 0.6, ((1, 0), (1, 0)): 0.3, ((0, 1), (1, 0)): 0.1j, ((1, 0), (0, 1)): -0.1j}
        extra = [((0, 2), (0, 0), 1.0), ((1, 0), (0, 1), 0.5j)]
    else:
        p = configs.kerr_driven(N=6, dt=0.002, T=18 * 0.002)
        extra = [((1,), (0,), 0.4 + 0.3j)]
        p.rho0 = {((0,), (0,)): 0.6, ((1,), (1,)): 0.4, ((0,), (1,)): 0.1j, ((1,), (0,)): -0.1j}
    q = len(p.params)
    p.h_terms = list(p.h_terms) + [HTerm(0.3, (1,) + (0,) * (modes - 1), (1,) + (0,) * (modes - 1), param=q)]
    for u, v, c in extra:
        p.h_terms += [HTerm(c, u, v, param=q), HTerm(complex(c).conjugate(), v, u, param=q)]
    p.params = list(p.params) + [0.0]
    loss, gt, gp = ograd.loss_and_grad(p, checkpoint_every=8)
    ref = np.concatenate([gt] + [gp[c].reshape(-1) for c in sorted(gp)])
    assert abs(gt[q]) > 1e-6
    for kw in (dict(resident=1), dict(resident=0), dict(resident=0, grad_coop=0)):
        st = gpu_state(p)
        st.set_tune(**kw)
        l, g = st.grad(p.dt, p.n_steps, 8)
        assert abs(l[0] - loss) <= 1e-12 * max(1.0, abs(loss))
        assert np.max(np.abs(g - ref)) <= 1e-10 * np.max(np.abs(ref)), kw


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_frequencies_that_cancel_cancel_exactly(dtype):
    """Three equal uncoupled oscillators in the lab frame: between permutations of the same occupation numbers
    the frequencies cancel, and such elements of A do not change (rounded sums over the modes differ with
    the order: the test takes the permutations where they do)."""
    N, w, eta = 5, 20.1, 1.3
    unit = lambda j, x: tuple(x if i == j else 0 for i in range(3))  # noqa: E731
    d = [(np.float64 if dtype == "f64" else np.float32)(w * k + eta * k * (k - 1)) for k in range(N)]
    meas = {}
    for k in itertools.permutations(range(N), 3):
        if d[k[0]] + d[k[1]] + d[k[2]] != d[k[1]] + d[k[2]] + d[k[0]]:
            meas[(k, k[1:] + k[:1])] = 1.0 + 0.5j
    assert meas
    h = [HTerm(w, unit(j, 1), unit(j, 1)) for j in range(3)] + [HTerm(eta, unit(j, 2), unit(j, 2)) for j in range(3)]
    q = configs.table_one_network(3, N, steps=4000)
    p = dataclasses.replace(q, h_terms=h, channels=[], secular=[], jumps=[], measured=meas, T=40 * q.dt)
    st = gpu_state(p, dtype=dtype, method="direct")
    assert st.get_tune()["resident"] == 1
    before = _raw(st, dtype)
    st.step(p.dt, 40)
    assert np.array_equal(_raw(st, dtype), before)


@pytest.mark.parametrize("modes,N", [(3, 5), (3, 6), (4, 4)])
def test_states_without_R_count_the_points_they_hold(modes, N):
    """R = 0: 64 to 125 systems of G_x and G_y alone (three modes at N = 6: 54 000 points, 5.8 million if R
    were stored) take the grid kernel."""
    p = configs.table_one_network(modes, N, steps=4000)
    a, b = _both(dataclasses.replace(p, T=12 * p.dt), "f64", 12, r_layout="off")
    _agree(a, b, "f64")


@pytest.mark.parametrize("instances,N,entries", [(1, 8, 4), (1, 8, 64), (25, 9, 4), (100, 8, 4), (40, 40, 4)])
def test_few_problems_of_several_initial_conditions(instances, N, entries):
    """One-mode FP64 problems whose measured operator has several entries (a system each), on both sides of
    what the grid kernels hold (40 problems of four at N = 40 stay with the resident kernel)."""
    meas = {((i % 8,), (i // 8,)): 1.0 / (1 + i) + 0.1j for i in range(entries)}
    ps = [dataclasses.replace(configs.kerr_driven(N=N, dt=0.002, T=0.05, n_th=0.1), measured=meas) for _ in range(instances)]
    a, b = gpu_state(ps, dtype="f64"), gpu_state(ps, dtype="f64")
    b.set_tune(resident=0)
    for n in (1, 13):
        a.step(ps[0].dt, n)
        b.step(ps[0].dt, n)
    _agree(a, b, "f64")
