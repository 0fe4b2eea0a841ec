"""Path updates of harmonic systems (ho_update.cu) against the pieces of the update,
pamd_mala_propose -> pamd_action_grad -> reverse -> accept -> commit, which run the
separate kernels: bit for bit, at the edges of element blocks (4096 elements), vectors
(chains that start off 16 bytes) and slice sizes, with rejected and accepted proposals."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pamd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1907_09529_gb300 as m
    m.tune()
    return m


# systems as (N, d, T, chains)
SHAPES = [
    [(1, 1, 1, 3)], [(1, 1, 2, 2)], [(1, 3, 1, 5)], [(1, 1, 1023, 3)],
    [(1, 1, 4094, 2)], [(1, 1, 4095, 3)], [(1, 1, 4096, 3)], [(1, 3, 1364, 3)], [(1, 3, 1365, 3)],
    [(1, 2, 4100, 3)], [(1, 3, 5003, 3)], [(4, 1, 2048, 2)], [(5, 1, 1700, 3)], [(2, 3, 700, 2)],
    [(21, 3, 130, 3)], [(64, 1, 63, 2)], [(64, 1, 64, 2)], [(65, 1, 80, 2)],
    [(1, 1, 700, 2), (1, 3, 301, 3), (5, 1, 99, 1)], [(1, 1, 700, 2), (1, 3, 3001, 3), (5, 1, 99, 1)],
]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "+".join("x".join(map(str, q)) for q in s))
def test_update_equals_its_pieces(pamd, shape, precision):
    dt, n = 0.02, 4
    prob = pamd.Problem([pamd.System("harmonic", N, d, T, B, k=0.8 + 0.1 * q)
                         for q, (N, d, T, B) in enumerate(shape)], 0.9, 1.1, dt, precision)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(len(shape) * 1000 + prob.span)
    pos = prob.empty("cuda")
    for q in range(len(shape)):
        v = prob.view(pos, q)
        v.copy_((torch.randn(v.shape, generator=gen, device="cuda") * (2 * 0.9 * dt) ** 0.5).cumsum(1))
    # a step at which proposals are accepted about half of the time
    h = 0.9 * dt * max(T * d * N for N, d, T, B in shape) ** (-1.0 / 3.0)
    S, g = pamd.action_grad(prob, pos)
    nacc = torch.zeros(prob.n_chains, dtype=torch.int32, device="cuda")
    p1, g1, S1, n1 = pos.clone(), g.clone(), S.clone(), nacc.clone()
    la = torch.zeros(prob.n_chains, dtype=torch.float64, device="cuda")
    la1 = la.clone()
    for u in range(n):  # the pieces
        prop, qf = pamd.mala_propose(prob, p1, g1, h, seed=5, counter=40 + u)
        Sp, gp = pamd.action_grad(prob, prop)
        qr = pamd.mala_reverse(prob, p1, prop, gp, h)
        acc = pamd.mala_accept(prob, S1, Sp, qf, qr, h, seed=5, counter=40 + u, n_accepted=n1, log_alpha=la1)
        pamd.mala_commit(prob, p1, g1, S1, prop, gp, Sp, acc)
    pamd.path_update(prob, pos, g, S, h, n, seed=5, counter=40, n_accepted=nacc, log_alpha=la)
    torch.cuda.synchronize()
    for a, b in ((pos, p1), (S, S1), (nacc, n1), (la, la1)):
        assert torch.equal(a, b)
    for q in range(len(shape)):
        assert torch.equal(prob.view(g, q), prob.view(g1, q))


@pytest.mark.parametrize("n,first", [(64, 1), (65, 64), (130, 63)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_updates_of_one_call_equal_those_of_two(pamd, precision, n, first):
    """Calls longer than one batch of uniforms."""
    dt = 0.02
    prob = pamd.Problem([pamd.System("harmonic", 1, 1, 600, 3, k=0.8)], 0.9, 1.1, dt, precision)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    pos = prob.empty("cuda")
    v = prob.view(pos, 0)
    v.copy_((torch.randn(v.shape, generator=gen, device="cuda") * (2 * 0.9 * dt) ** 0.5).cumsum(1))
    h = 0.9 * dt * 600 ** (-1.0 / 3.0)
    S, g = pamd.action_grad(prob, pos)
    out = []
    for parts in ([n], [first, n - first]):
        p1, g1, S1 = pos.clone(), g.clone(), S.clone()
        nacc = torch.zeros(prob.n_chains, dtype=torch.int32, device="cuda")
        la = torch.zeros(prob.n_chains, dtype=torch.float64, device="cuda")
        at = 7
        for m in parts:
            pamd.path_update(prob, p1, g1, S1, h, m, seed=5, counter=at, n_accepted=nacc, log_alpha=la)
            at += m
        out.append((p1, prob.view(g1, 0).clone(), S1, nacc, la))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    assert 0 < int(out[0][3].min()) and int(out[0][3].max()) < n
