"""How a batch is cut into work items (pamd_api.cu) changes the order of the FP64 sums of S
and nothing else: the automatic cut against items of 32 steps, where the rule turns --
chains of one step, fewer steps than CTAs, a few more steps than CTAs, many short chains
(more rounds of shorter items), unlike systems, both block-size classes."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import pamd_inputs as inputs  # noqa: E402


@pytest.fixture(scope="module")
def pamd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1907_09529_gb300 as m
    m.tune()
    return m


@pytest.mark.parametrize("shape", [
    [(64, 1, 3)], [(108, 30, 5)], [(600, 77, 2)], [(108, 31, 64)], [(100, 130, 40)], [(700, 40, 9)],
    [(64, 5, 1), (108, 300, 2), (256, 90, 3), (500, 61, 1)], [(108, 400, 2), (600, 50, 3), (860, 1, 1)],
], ids=lambda s: "+".join("x".join(map(str, q)) for q in s))
def test_automatic_items_equal_items_of_32_steps(pamd, shape):
    systems = []
    for N, T, B in shape:
        L = inputs.box_side(N, 0.85)
        systems.append(pamd.System("lj", N, 3, T, B, box=L, rc=min(2.5, L / 2)))
    prob = pamd.Problem(systems, 1.0, 1.0, 1e-4)
    pos = prob.empty("cuda")
    for q, (N, T, B) in enumerate(shape):
        x0 = torch.from_numpy(inputs.fcc_lattice(N, systems[q].box)).float().cuda()
        gen = torch.Generator(device="cuda")
        gen.manual_seed(N)
        v = prob.view(pos, q)
        step = torch.randn(v.shape, generator=gen, device="cuda") * 0.01
        v.copy_(x0 + step.cumsum(1) * (step.shape[1] < 100) + step)
    try:
        S, g = pamd.action_grad(prob, pos)
        S1 = pamd.action(prob, pos)
        pamd.tune(32)
        S32, g32 = pamd.action_grad(prob, pos)
    finally:
        pamd.tune()
    torch.cuda.synchronize()
    for q in range(len(shape)):
        assert torch.equal(prob.view(g, q), prob.view(g32, q))
    # sums of at most 300 items a chain in FP64
    for a in (S, S1):
        assert float(((a - S32).abs() / S32.abs()).max()) < 1e-13


@pytest.mark.parametrize("shapes", [[(64, 2001, 8)], [(600, 2503, 4)], [(96, 1777, 5), (560, 1333, 6)]])
def test_parts_of_long_items(pamd, shapes):
    """Items of several parts (device buffers) and the parts as items of their own (chunks of
    chains in the host-buffer pipeline): the same action, update and acceptance, bit for bit."""
    systems = []
    for N, T, B in shapes:
        L = inputs.box_side(max(N, 108), 0.85)
        systems.append(pamd.System("lj", N, 3, T, B, box=L, rc=2.3))
    prob = pamd.Problem(systems, 1.0, 1.0, 1e-4)
    buf = prob.empty("cuda")
    for q, s in enumerate(systems):
        prob.view(buf, q)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(s.N, s.box)))
    pamd.euler_reference(prob, buf, seed=6)
    S, g = pamd.action_grad(prob, buf)
    assert torch.equal(S, pamd.action(prob, buf))
    host = [t.cpu() for t in (buf, g, S)]
    nacc = [torch.zeros(prob.n_chains, dtype=torch.int32, device=d) for d in ("cuda", "cpu")]
    la = [torch.zeros(prob.n_chains, dtype=torch.float64, device=d) for d in ("cuda", "cpu")]
    h = 2e-7
    pamd.path_update(prob, buf, g, S, h, 2, seed=3, n_accepted=nacc[0], log_alpha=la[0])
    pamd.path_update(prob, *host, h, 2, seed=3, n_accepted=nacc[1], log_alpha=la[1])
    torch.cuda.synchronize()
    assert torch.equal(nacc[0].cpu(), nacc[1]) and torch.equal(la[0].cpu(), la[1])
    assert torch.equal(S.cpu(), host[2])
    for q in range(len(systems)):
        assert torch.equal(prob.view(buf, q).cpu(), prob.view(host[0], q))
        assert torch.equal(prob.view(g, q).cpu(), prob.view(host[1], q))


@pytest.mark.parametrize("N,B", [(520, 1), (560, 3), (700, 2), (300, 2), (90, 3), (33, 4)])
def test_overflowing_lists_give_the_same_results(pamd, N, B):
    """Window lists that overflow (all of them, with room for a few entries) take their
    candidates from the outer lists, or from all particles where these are not much shorter:
    bit for bit the results of lists with room, for long and short items."""
    T, L = 70, inputs.box_side(864, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4)
    pos = prob.empty("cuda")
    prob.view(pos, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(864, L)[:, :N].copy()))
    pamd.euler_reference(prob, pos, seed=2)
    out = []
    try:
        for tile, cap in ((0, 0), (0, 24), (7, 24), (0, 1)):
            pamd.tune(tile, 0, cap)
            S, g = pamd.action_grad(prob, pos)
            assert torch.equal(S, pamd.action(prob, pos))
            out.append((S.clone(), prob.view(g, 0).clone()))
    finally:
        pamd.tune()
    torch.cuda.synchronize()
    for S, g in out[1:]:
        assert torch.equal(g, out[0][1])
        assert float(((S - out[0][0]).abs() / S.abs()).max()) < 1e-13  # FP64 sums of the items
