"""Waits between the CTAs of a cluster that run out (PAMD_FAULT_INJECT=wait:N: the odd CTAs
leave after N rounds, and waits last two milliseconds).  The call ends and leaves
PAMD_ERR_TIMEOUT, a path that could not be finished is NaN and an update that could not be
finished changes nothing, and the next call is right.  The kernels wait for their stores in
flight before they end; a wait for one that never comes takes four seconds, which the time
limit here would show.  Nothing faults on the device."""
import os
import time

import pytest

import pamd_inputs as inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TIMEOUT = -4


@pytest.fixture(scope="module")
def pamd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1907_09529_gb300 as m
    m.tune()
    return m


@pytest.fixture
def fault():
    def set_(what):
        if what:
            os.environ["PAMD_FAULT_INJECT"] = what
        else:
            os.environ.pop("PAMD_FAULT_INJECT", None)
    yield set_
    os.environ.pop("PAMD_FAULT_INJECT", None)


def _times_out(pamd, call):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    call()
    with pytest.raises(pamd.PamdError) as ei:
        pamd.device_status()
    assert ei.value.status == TIMEOUT and time.perf_counter() - t0 < 1.5
    pamd.device_status()  # cleared


# all pairs with 2, 4 and 8 CTAs, in order and packed, and lists
@pytest.mark.parametrize("precision,N,B", [("fp32", 57, 1), ("fp32", 108, 4), ("fp32", 150, 25), ("fp32", 193, 1),
                                           ("fp32", 500, 30), ("fp64", 33, 2), ("fp64", 64, 60), ("fp64", 108, 3),
                                           ("fp64", 250, 2)])
def test_euler_path(pamd, fault, precision, N, B):
    T, L = 30, inputs.box_side(512, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4, precision)
    start = torch.zeros(prob.span + 64, dtype=prob.dtype, device="cuda")  # with a guard behind
    prob.view(start, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(512, L)[:, :N].copy()))
    want = start.clone()
    pamd.euler_reference(prob, want, seed=3, counter=1)
    pamd.device_status()
    for first in (1, 2, 3, 12, T - 1):
        buf = start.clone()
        fault("wait:%d" % first)
        _times_out(pamd, lambda: pamd.euler_reference(prob, buf, seed=3, counter=1))
        fault(None)
        v = prob.view(buf, 0)
        assert torch.equal(v[:, 0], prob.view(start, 0)[:, 0]) and bool(torch.isnan(v[:, 1:]).all())
        assert not bool(buf[prob.span:].any())
    buf = start.clone()
    pamd.euler_reference(prob, buf, seed=3, counter=1)
    pamd.device_status()
    assert torch.equal(prob.view(buf, 0), prob.view(want, 0))


@pytest.mark.parametrize("d,T,B", [(1, 1023, 1), (1, 250, 3), (3, 200, 30), (1, 1500, 19), (16, 60, 2), (1, 300, 76)])
def test_updates(pamd, fault, d, T, B):
    """Paths on 2, 4 and 8 CTAs: the state stays as it was."""
    n, dt = 9, 0.02
    prob = pamd.Problem([pamd.System("harmonic", d if d == 16 else 1, 1 if d == 16 else d, T, B, k=0.8)], 0.9, 1.1, dt,
                        "fp64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    pos = prob.empty("cuda")
    v = prob.view(pos, 0)
    v.copy_((torch.randn(v.shape, generator=gen, device="cuda") * (2 * 0.9 * dt) ** 0.5).cumsum(1))
    S, g = pamd.action_grad(prob, pos)
    h = 0.9 * dt * (T * d) ** (-1.0 / 3.0)

    def state():
        return [pos.clone(), g.clone(), S.clone(), torch.zeros(B, dtype=torch.int32, device="cuda"),
                torch.full((B,), 7.0, dtype=torch.float64, device="cuda")]

    def update(s):
        pamd.path_update(prob, s[0], s[1], s[2], h, n, seed=5, counter=40, n_accepted=s[3], log_alpha=s[4])

    def same(a, b):
        for q in range(2):
            assert torch.equal(prob.view(a[q], 0), prob.view(b[q], 0))
        for q in range(2, 5):
            assert torch.equal(a[q], b[q])

    want = state()
    update(want)
    pamd.device_status()
    for first in (0, 1, 2, 5, n - 1):
        s = state()
        fault("wait:%d" % first)
        _times_out(pamd, lambda: update(s))
        fault(None)
        same(s, state())
    s = state()
    update(s)
    pamd.device_status()
    same(s, want)


def test_host_buffers_get_the_status(pamd, fault):
    """Calls with host buffers return it themselves, and it is cleared."""
    N, T, B, L = 108, 20, 2, inputs.box_side(108, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.3)], 1.0, 1.0, 1e-4, "fp64")
    buf = prob.empty("cpu")
    prob.view(buf, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(N, L)))
    fault("wait:3")
    with pytest.raises(pamd.PamdError) as ei:
        pamd.euler_reference(prob, buf, seed=3, counter=1)
    assert ei.value.status == TIMEOUT
    fault(None)
    pamd.device_status()
    pamd.euler_reference(prob, buf, seed=3, counter=1)
    assert bool(torch.isfinite(prob.view(buf, 0)).all())
    for chains in (1, 3):  # one stream, and the pipeline over chunks
        ho = pamd.Problem([pamd.System("harmonic", 1, 1, 500, chains, k=0.8)], 0.9, 1.1, 0.02, "fp64")
        pos = 0.1 * torch.randn(ho.span, dtype=torch.float64)
        S, g = torch.zeros(chains, dtype=torch.float64), torch.zeros(ho.span, dtype=torch.float64)
        pamd.action_grad(ho, pos, S, g)
        before = [t.clone() for t in (pos, g, S)]
        nacc = torch.zeros(chains, dtype=torch.int32)
        fault("wait:0")
        with pytest.raises(pamd.PamdError) as ei:
            pamd.path_update(ho, pos, g, S, 1e-6, 4, seed=1, n_accepted=nacc)
        assert ei.value.status == TIMEOUT
        fault(None)
        pamd.device_status()
        assert all(torch.equal(a, b) for a, b in zip((pos, g, S), before))
        pamd.path_update(ho, pos, g, S, 1e-6, 4, seed=1, n_accepted=nacc)
        pamd.device_status()
        assert int(nacc.min()) > 0


def test_a_later_status_does_not_replace_it(pamd, fault):
    prob = pamd.Problem([pamd.System("harmonic", 1, 1, 500, 1, k=0.8)], 0.9, 1.1, 0.02, "fp64")
    pos = prob.empty("cuda")
    prob.view(pos, 0).zero_()
    S, g = pamd.action_grad(prob, pos)
    pamd.device_status()
    fault("wait:0")
    pamd.path_update(prob, pos, g, S, 1e-6, 4, seed=1)
    fault(None)
    prob.view(pos, 0)[0, 3] = float("nan")
    pamd.action_grad(prob, pos)  # a non-finite action
    with pytest.raises(pamd.PamdError) as ei:
        pamd.device_status()
    assert ei.value.status == TIMEOUT
    pamd.action_grad(prob, pos)
    with pytest.raises(pamd.PamdError) as ei:
        pamd.device_status()
    assert ei.value.status == -5  # PAMD_ERR_NONFINITE
