"""Error paths, exercised by host-side fault injection (PAMD_FAULT_INJECT): the
documented status comes back, nothing half-built stays cached, and the library
works normally once the fault is gone.  Nothing faults on the device."""
import os

import pytest

import pamd_inputs as inputs
from _common import gpu_system, start_paths

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pamd():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_1907_09529_gb300 as pamd
    pamd.tune()
    return pamd


@pytest.fixture
def fault():
    def set_(what):
        if what:
            os.environ["PAMD_FAULT_INJECT"] = what
        else:
            os.environ.pop("PAMD_FAULT_INJECT", None)
    yield set_
    os.environ.pop("PAMD_FAULT_INJECT", None)


def _case(pamd):
    w = inputs.workload("lj108", "small")
    prob = pamd.Problem([gpu_system(s, pamd) for s in w.systems], w.D, w.beta, w.dt)
    buf = prob.empty("cuda")
    for q, p in enumerate(start_paths(w, "fp32")):
        prob.view(buf, q).copy_(torch.from_numpy(p).float())
    return prob, buf


def test_allocation_failure_leaves_no_plan(pamd, fault):
    prob, buf = _case(pamd)
    pamd.release_cache()
    fault("alloc")
    with pytest.raises(pamd.PamdError) as ei:
        pamd.action_grad(prob, buf)
    assert ei.value.status == -6  # PAMD_ERR_ALLOC
    assert pamd.cache_stats() == (0, 0)
    fault(None)
    S, g = pamd.action_grad(prob, buf)
    torch.cuda.synchronize()
    assert pamd.cache_stats() == (1, 0) and bool(torch.isfinite(S).all())


def test_cuda_failure_is_reported_and_recovers(pamd, fault):
    prob, buf = _case(pamd)
    pamd.release_cache()
    S0, g0 = pamd.action_grad(prob, buf)  # plan built and cached
    torch.cuda.synchronize()
    fault("launch")
    with pytest.raises(pamd.PamdError) as ei:
        pamd.action_grad(prob, buf)
    assert ei.value.status == -3  # PAMD_ERR_CUDA
    nacc = torch.zeros(prob.n_chains, dtype=torch.int32, device="cuda")
    with pytest.raises(pamd.PamdError) as ei:  # a capture that fails caches no graph
        pamd.path_update(prob, buf, g0.clone(), S0.clone(), 1e-6, n_updates=3, n_accepted=nacc)
    assert ei.value.status == -3
    assert pamd.cache_stats() == (1, 0)
    fault(None)
    S1, g1 = pamd.action_grad(prob, buf)
    torch.cuda.synchronize()
    assert torch.equal(S1, S0) and torch.equal(g1, g0)
    pamd.path_update(prob, buf, g1, S1, 1e-6, n_updates=3, n_accepted=nacc)
    torch.cuda.synchronize()
    assert pamd.cache_stats() == (1, 1)


def test_nonfinite_flag_is_reported_once(pamd, fault):
    prob, buf = _case(pamd)
    pamd.device_status()  # clear anything earlier
    fault("nonfinite")
    pamd.action_grad(prob, buf)
    fault(None)
    with pytest.raises(pamd.PamdError) as ei:
        pamd.device_status()
    assert ei.value.status == -5  # PAMD_ERR_NONFINITE
    pamd.device_status()  # cleared
    pamd.action_grad(prob, buf)
    pamd.device_status()  # a clean call reports nothing


@pytest.mark.parametrize("precision,limit", [("fp32", 1 << 21), ("fp32", 1 << 19), ("fp64", 1 << 26), ("fp64", 1 << 24)])
def test_less_scratch_gives_the_same_results(pamd, fault, precision, limit):
    """Neighbour lists and pair records that do not fit the device become shorter, and the
    host-buffer pipeline runs with the lanes it has scratch for; the results stay."""
    N, T, B, L = 200, 160, 4, inputs.box_side(256, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4, precision)
    buf = prob.empty("cuda")
    prob.view(buf, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(256, L)[:, :N].copy()))
    pamd.euler_reference(prob, buf, seed=4)

    def update():
        host = [t.cpu() for t in (buf, g, S)]
        pamd.path_update(prob, *host, 1e-7, 2, seed=3)
        return host

    pamd.release_cache()
    S, g = pamd.action_grad(prob, buf)
    want = update()
    pamd.release_cache()
    fault("alloc:%d" % limit)
    S1, g1 = pamd.action_grad(prob, buf)
    torch.cuda.synchronize()
    assert torch.equal(S, S1) and torch.equal(prob.view(g, 0), prob.view(g1, 0))
    fault(None)  # the plan has its short lists; the staging buffers fit, two more lanes do not
    pamd.action_grad(prob, buf.cpu())
    got = update()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    pamd.release_cache()


def test_pipeline_without_scratch_for_its_lanes(pamd, fault):
    N, T, B, L = 200, 160, 4, inputs.box_side(256, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4, "fp64")
    buf = prob.empty("cuda")
    prob.view(buf, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(256, L)[:, :N].copy()))
    pamd.euler_reference(prob, buf, seed=4)
    out = []
    for limit in (None, "alloc:%d" % (1 << 24)):  # (the path takes 3.1 MB, a lane's scratch 110 MB)
        pamd.release_cache()
        S, g = pamd.action_grad(prob, buf)  # lane 0's scratch
        host = [t.cpu() for t in (buf, g, S)]
        fault(limit)
        pamd.path_update(prob, *host, 1e-7, 2, seed=3)
        fault(None)
        out.append(host)
    assert all(torch.equal(a, b) for a, b in zip(*out))
    pamd.release_cache()


def test_device_memory_of_a_plan(pamd):
    """A plan that the host-buffer pipeline has not used holds one lane's lists: about 70 MB
    for 500 particles on 152 SMs, not three times that."""
    L = inputs.box_side(500, 0.85)
    small = pamd.Problem([pamd.System("lj", 500, 3, 16, 1, box=L, rc=2.5)], 1.0, 1.0, 1e-4)
    prob = pamd.Problem([pamd.System("lj", 500, 3, 4096, 8, box=L, rc=2.5)], 1.0, 1.0, 1e-4)
    buf, sbuf = torch.zeros(prob.span, device="cuda"), torch.zeros(small.span, device="cuda")
    for p, b in ((small, sbuf), (prob, buf)):
        p.view(b, 0)[:] = torch.from_numpy(inputs.fcc_lattice(500, L)).float()[None, None].cuda()
    pamd.release_cache()
    pamd.action(small, sbuf)
    S = torch.empty(8, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    pamd.action(prob, buf, S)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    pamd.release_cache()
    assert used < 100 << 20
