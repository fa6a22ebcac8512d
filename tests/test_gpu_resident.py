"""The resident single-mode kernel (whole steps on chip; bq_tune resident = 1) against the
streaming kernels (resident = 0) and the oracle: grid sizes at the edges of its strips, both
layouts (Hermitian systems, general ones), every form of term and envelope it takes, and the
forms it must leave to the other kernels."""

import dataclasses

import numpy as np
import pytest

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


def _problem(N, n_th=0.05, drive="gauss", measured=None, steps=11, secular=False):
    p = configs.kerr_driven(N=N, dt=0.002, T=steps * 0.002, n_th=n_th)
    T = p.T
    kinds = {"gauss": Channel("gauss", (0.3, 0.0, 0.4 * T, 0.3 * T)), "gauss_complex": Channel("gauss", (0.3, 0.2, 0.4 * T, 0.3 * T)),
             "pwc": Channel("pwc", (0.0, T / 3.0, 0.3, 0.1, -0.2, 0.2, 0.1, -0.1)), "cexp": Channel("cexp", (0.3, -0.1, 2.0)),
             "const": Channel("const", (0.2, 0.0))}
    if drive is None:
        p.h_terms = [t for t in p.h_terms if t.channel < 0]
        p.channels = []
    else:
        p.channels = [kinds[drive]]
    if measured is not None:
        p.measured = measured
    if secular:
        p.jumps = []
        p.secular = [SecularDamping(0, 0.05, (0.1,) * (N - 1) if n_th else ())]
    return p


GENERAL = {((0,), (1,)): 1.0 + 0.5j, ((2,), (2,)): 0.7, ((1,), (0,)): 0.2j}  # p != q: the general layout
SIZES = (4, 5, 7, 8, 13, 14, 16, 17, 24, 25, 32, 33, 37, 40, 41, 42)


def _both(ps, dtype, steps, **kw):
    a, b = gpu_state(ps, dtype=dtype, **kw), gpu_state(ps, dtype=dtype, **kw)
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    a.step(ps[0].dt, steps)
    b.step(ps[0].dt, steps)
    return a, b


def _agree(a, b, dtype):
    x, y = _raw(a, dtype), _raw(b, dtype)
    assert np.all(np.isfinite(x))
    assert np.max(np.abs(x - y)) <= TOL[dtype] * np.max(np.abs(y))
    ea, eb = a.evaluate(), b.evaluate()
    assert np.max(np.abs(ea - eb)) <= TOL[dtype] * max(1.0, np.max(np.abs(eb)))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("measured", [None, GENERAL])
def test_every_grid_size_matches_streaming_and_oracle(dtype, measured):
    ps = [_problem(N, measured=measured) for N in SIZES]
    a, b = _both(ps, dtype, 11)
    _agree(a, b, dtype)
    off = 0
    for p in ps:
        n = len(p.measured)
        if p.N[0] in (4, 17, 42):
            compare_mapped_systems(a, mapping.rk4_mapped(p), 1e-10 if dtype == "f64" else 1e-5, sys_offset=off, n_sys=off + n)
        off += n


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("measured", [None, GENERAL])
@pytest.mark.parametrize("form", [dict(drive="gauss_complex"), dict(drive="pwc"), dict(drive="cexp"), dict(drive="const"),
                                  dict(drive=None), dict(n_th=0.0), dict(secular=True), dict(secular=True, n_th=0.0)])
@pytest.mark.parametrize("reverse", [True, False])
def test_every_form_matches_streaming(dtype, measured, form, reverse):
    ps = [dataclasses.replace(_problem(N, measured=measured, **form), reverse_time=reverse) for N in (5, 12, 31, 40)]
    a, b = _both(ps, dtype, 11)
    _agree(a, b, dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("measured", [None, GENERAL])
def test_direct_method_and_solve(dtype, measured):
    ps = [_problem(N, measured=measured) for N in (6, 21, 40)]
    a, b = _both(ps, dtype, 9, method="direct")
    _agree(a, b, dtype)
    c = gpu_state(ps, dtype=dtype, method="direct")
    c.solve(ps[0].dt, 9)
    assert np.array_equal(_raw(c, dtype), _raw(a, dtype))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_loaded_states_take_the_layout_their_data_need(dtype):
    """After bq_load_state the data decide: the Hermitian state of the same run continues bit for
    bit; a state that is not Hermitian is stepped in the general layout; stepping by the other
    kernels in between is followed."""
    import torch
    ps = [_problem(N) for N in (6, 13, 40)]
    ft = torch.float64 if dtype == "f64" else torch.float32
    a, b = _both(ps, dtype, 7)
    snap = torch.from_numpy(_raw(a, dtype)).to(ft)
    gen = torch.Generator().manual_seed(5)
    noisy = (snap + 1e-2 * torch.randn(snap.shape, generator=gen, dtype=torch.float64)).to(ft)
    # the padding of the blocks is zero in every state
    clean = gpu_state(ps, dtype=dtype)
    info = [clean.system_info(i) for i in range(3)]
    keep, off = torch.zeros_like(snap), 0
    for s in info:
        for n in (s["n_gx"], s["n_gy"], s["n_r"]):
            keep[2 * off:2 * (off + n)] = 1
            off += (n + 3) & ~3
    for data in (snap, noisy * keep):
        host = data.contiguous().pin_memory()
        x, y = gpu_state(ps, dtype=dtype), gpu_state(ps, dtype=dtype)
        y.set_tune(resident=0)
        for st in (x, y):
            st.load_state(host.data_ptr())
            st.step(ps[0].dt, 3)
            st.step(ps[0].dt, 2)
        _agree(x, y, dtype)
    x.set_tune(resident=0)
    x.step(ps[0].dt, 2)
    x.set_tune(resident=1)
    x.step(ps[0].dt, 2)
    y.step(ps[0].dt, 4)
    _agree(x, y, dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_calls_split_anywhere_give_the_same_bits(dtype):
    ps = [_problem(N, drive="gauss_complex") for N in (5, 16, 33)]
    a, b = gpu_state(ps, dtype=dtype), gpu_state(ps, dtype=dtype)
    a.step(ps[0].dt, 33)
    for n in (1, 8, 7, 16, 1):
        b.step(ps[0].dt, n)
    assert np.array_equal(_raw(a, dtype), _raw(b, dtype))
    assert np.array_equal(a.evaluate(), b.evaluate())


def test_other_forms_keep_the_other_kernels():
    def one(f):
        p = _problem(9)
        f(p)
        st = gpu_state(p)
        st.set_tune(resident=1)
        return st.get_tune()["resident"]

    a, a2, z = (1,), (2,), (0,)
    assert one(lambda p: None) == 1
    assert one(lambda p: p.h_terms.extend([HTerm(0.2, a2, z), HTerm(0.2, z, a2)])) == 0  # shift 2
    assert one(lambda p: p.h_terms.append(HTerm(0.2, a, a, channel=0)) or p.h_terms.append(HTerm(0.2, a, a, channel=0, conj=True))) == 0
    assert one(lambda p: p.h_terms.extend([HTerm(0.1, a, z), HTerm(0.1, z, a)])) == 0  # two drives
    assert one(lambda p: p.jumps.append(Jump(0.1, ((1.0 + 0j, a, a),)))) == 0  # dephasing: shift 0
    assert one(lambda p: p.jumps.append(Jump(0.1, ((1.0 + 0j, z, a), (0.5 + 0j, z, z))))) == 0  # L = a + 1/2
    assert gpu_state(_problem(43)).get_tune()["resident"] == 0
    assert gpu_state(_problem(3, measured={((1,), (1,)): 1.0})).get_tune()["resident"] == 0
    assert gpu_state(_problem(9), r_layout="off").get_tune()["resident"] == 0
    assert gpu_state([_problem(9), _problem(43)]).get_tune()["resident"] == 0  # one problem decides for the batch


def test_replayed_graphs_leave_no_stale_observables():
    """bq_step on the one-CTA-per-system kernel (the second call of 64 steps replays its graph) with a
    resident solve in between: the observables, and the next solve, are those of the current state.
    (dt: FP32 phases of the highest level stay at O(1) rad, as the tolerance assumes.)"""
    ps, dt = [_problem(N, steps=200) for N in (6, 13, 16)], 2e-4
    a, b = gpu_state(ps, dtype="f32"), gpu_state(ps, dtype="f32")
    a.set_tune(stage_path="system")
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    a.step(dt, 64)
    b.step(dt, 64)
    a.solve(dt, 5)
    b.step(dt, 5)
    before = a.evaluate()
    a.step(dt, 64)
    b.step(dt, 64)
    assert not np.array_equal(a.evaluate(), before)
    _agree(a, b, "f32")
    a.solve(dt, 5)
    b.step(dt, 5)
    _agree(a, b, "f32")


@pytest.mark.parametrize("measured", [None, GENERAL])
@pytest.mark.parametrize("instances", [1, 200])
def test_fp64_update_keeps_the_bits_of_elements_below_their_increment(instances, measured):
    """A step's update is error-free in FP64 as on the streaming kernels, also where the increment is the
    larger operand: elements of 2^-100 with increments above 2^-40 are left as the sum's residual.  One
    system (the grid kernel) and 200 (the resident kernel)."""
    import torch
    ps = [_problem(24, measured=measured) for _ in range(instances)]
    a, b = gpu_state(ps, dtype="f64"), gpu_state(ps, dtype="f64")
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    eps, n = 2.0 ** -100, 24
    info = [a.system_info(i) for i in range(a.n_systems())]
    host = torch.zeros(a.state_bytes() // 16, dtype=torch.complex128)
    rng, off, small = np.random.default_rng(3), 0, []
    for s in info:
        z = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
        z = z + z.conj().T
        for i in range(0, n - 2, 3):
            z[i, i + 2] = z[i + 2, i] = eps
        g = rng.normal(size=n) + 1j * rng.normal(size=n)
        for v, m in ((g, s["n_gx"]), (g.conj(), s["n_gy"]), (z.reshape(-1), s["n_r"])):
            host[off:off + m] = torch.from_numpy(v)
            if m > n:
                small += [off + i * n + i + 2 for i in range(0, n - 2, 3)]
            off += (m + 3) & ~3
    host = host.pin_memory()

    def residual(st):
        """The rounding residual of the state, which follows the state in the pool."""
        st.load_state(host.data_ptr())
        st.step(ps[0].dt, 1)
        y = torch.empty(st.state_bytes(), dtype=torch.uint8, pin_memory=True)
        st.store_state(y.data_ptr())
        torch.cuda.synchronize()
        y, pool = y.numpy().tobytes(), st.pool.cpu().numpy().tobytes()
        at = pool.find(y)
        assert at >= 0
        at = (at + len(y) + 255) // 256 * 256
        return np.frombuffer(y, complex)[small], np.frombuffer(pool[at:at + len(y)], complex)[small]

    for st in (b, a):
        y, c = residual(st)
        assert np.min(np.abs(y.real)) > 2.0 ** -40
        assert np.all(c.real == -eps)


def test_a_gradient_that_fails_leaves_no_stale_observables():
    """Elements near the largest FP32 value overflow in a step and spread by at most four rows in each: the
    gradient is refused, and the observables afterwards are not those of the step before it."""
    import paper_2203_05526_gb300 as bq
    import torch
    p = _problem(14, steps=40)
    p.rho0 = {((0,), (0,)): 1.0}
    st = gpu_state(p, dtype="f32")
    assert st.get_tune()["resident"] == 1
    host = torch.zeros(st.state_bytes() // 8, dtype=torch.complex64)
    info = st.system_info(0)
    off = ((info["n_gx"] + 3) & ~3) + ((info["n_gy"] + 3) & ~3)
    host[off] = 1.0
    host[off + 12 * 14:off + 14 * 14] = 2.9e38 + 2.9e38j
    host = host.pin_memory()
    st.load_state(host.data_ptr())
    st.step(1e-9, 1)
    assert np.all(np.isfinite(st.evaluate()))
    with pytest.raises(bq.BQError):
        st.grad(p.dt, 16, 8)
    with pytest.raises(bq.BQError):
        st.evaluate()
