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
