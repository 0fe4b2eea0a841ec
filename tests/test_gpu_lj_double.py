"""Double-precision Lennard-Jones action and gradient (lj_double.cu) where it can go
wrong: row words of 32 particles and their remainders, one to eight threads per
particle, the largest N, particles in other periodic images, pairs beyond the record
capacity, items of one step, and cutoffs at half the box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import pamd_inputs as inputs  # noqa: E402
from _common import rel  # noqa: E402


@pytest.fixture(scope="module")
def pamd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1907_09529_gb300 as m
    m.tune()
    return m


def _check(pamd, N, T, B, L, rc, x0, tile=0, jitter=0.01, seed=1, tol=1e-12):
    """S and gradient of B paths jittering around x0 [3][N] against the oracle; the
    tolerance is the double-precision one of the parity tests."""
    D, beta, dt = 0.9, 1.1, 1e-4
    rng = inputs.rng(seed)
    walk = np.cumsum(jitter * rng.standard_normal((B, T + 1, 3, N)), axis=1)
    paths = x0[None, None] + walk
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=rc)], D, beta, dt, "fp64")
    buf = prob.empty("cuda")
    prob.view(buf, 0).copy_(torch.from_numpy(paths))
    try:
        pamd.tune(tile)
        S, g = pamd.action_grad(prob, buf)
        S1 = pamd.action(prob, buf)
        torch.cuda.synchronize()
    finally:
        pamd.tune()
    assert torch.equal(S, S1)
    pot = oracle.lennard_jones(L, rc)
    for b in range(B):
        So, go = oracle.action_grad(pot, paths[b], D, beta, dt, nthreads=8)
        gb = prob.view(g, 0)[b].cpu().numpy()
        assert abs(S[b].item() - So) <= tol * abs(So)
        assert rel(gb, go) <= tol
        assert np.abs(gb - go).max() <= tol * np.abs(go).max()
    return g


@pytest.mark.parametrize("N", [2, 3, 31, 32, 33, 63, 65, 127, 129, 257, 511, 513, 863, 1023, 1024])
def test_sizes(pamd, N):
    L = max(inputs.box_side(N, 0.85), 3.2)
    _check(pamd, N, 3, 2, L, min(2.5, L / 2), inputs.fcc_lattice(N, L), seed=N)


@pytest.mark.parametrize("T,tile", [(1, 0), (5, 1), (9, 4), (9, 0)])
def test_items(pamd, T, tile):
    L = inputs.box_side(64, 0.85)
    g = _check(pamd, 64, T, 3, L, L / 2, inputs.fcc_lattice(64, L), tile=tile, seed=4)
    assert torch.equal(g, _check(pamd, 64, T, 3, L, L / 2, inputs.fcc_lattice(64, L), tile=32, seed=4))


def test_other_images(pamd):
    """Particles stored up to 1000 boxes away: same forces as in the first box to the
    rounding of the stored coordinates (eps * 1000 L on distances, steep pair forces)."""
    N = 108
    L = inputs.box_side(N, 0.85)
    shift = inputs.rng(9).integers(-1000, 1001, size=(3, N)) * L
    _check(pamd, N, 4, 1, L, 2.5, inputs.fcc_lattice(N, L) + shift, seed=5)


def test_clustered_pairs_exceed_the_capacity(pamd):
    """A droplet in a large box holds far more pairs than the uniform density that the
    records are sized for."""
    N = 256
    x0 = inputs.fcc_lattice(N, inputs.box_side(N, 0.85))
    _check(pamd, N, 4, 2, 60.0, 2.5, x0, seed=6)


@pytest.mark.parametrize("boxes", [2 ** 20, 2 ** 30 - 1, 2 ** 30, 2 ** 31 + 5, 2 ** 33 - 2, 2 ** 40, 2 ** 43])
@pytest.mark.parametrize("tile", [0, 2])
def test_images_far_away(pamd, boxes, tile):
    """Every third particle stored some 2^20 to 2^43 box lengths away, as exploding paths
    are: box indices beyond 32 bits.  With a box of 8 every coordinate, difference and
    image is exact (multiples of 2^-5 below 2^48), so the tolerance is that of the parity tests."""
    N, L, T = 100, 8.0, 5
    x0 = inputs.fcc_lattice(N, L * 0.75)
    walk = 0.02 * inputs.rng(boxes % 1000).standard_normal((1, T + 1, 3, N)).cumsum(1)
    paths = np.round((x0 + walk) * 32.0) / 32.0
    paths[..., ::3] += boxes * L
    paths[:, :, 1, 1::3] -= boxes * L
    D, beta, dt = 0.9, 1.1, 1e-4
    prob = pamd.Problem([pamd.System("lj", N, 3, T, 1, box=L, rc=2.5)], D, beta, dt, "fp64")
    buf = prob.empty("cuda")
    prob.view(buf, 0).copy_(torch.from_numpy(paths))
    try:
        pamd.tune(tile)
        S, g = pamd.action_grad(prob, buf)
        S1 = pamd.action(prob, buf)
        torch.cuda.synchronize()
    finally:
        pamd.tune()
    So, go = oracle.action_grad(oracle.lennard_jones(L, 2.5), paths[0], D, beta, dt, nthreads=8)
    near = paths[0].copy()
    near[..., ::3] -= boxes * L
    near[:, 1, 1::3] += boxes * L
    Sn, gn = oracle.action_grad(oracle.lennard_jones(L, 2.5), near, D, beta, dt, nthreads=8)
    assert abs(So - Sn) <= 1e-12 * Sn and rel(go, gn) <= 1e-12  # (the oracle's images are exact too)
    assert torch.equal(S, S1) and abs(S[0].item() - So) <= 1e-12 * So
    assert rel(prob.view(g, 0)[0].cpu().numpy(), go) <= 1e-12


@pytest.mark.parametrize("k", [-58, -57, -56, -55, -54, -1, 1, 46, 47, 48, 49, 50])
def test_units_of_any_size(pamd, k):
    """Lengths in units of 2^k (energies of 4^k): every term scales by a power of two, but for
    1/r, which has a form of its own where r^2 lies in 2^-111..2^97 and the library's elsewhere.
    A few ulp of 1/r (2e-16 each) to the power 14 and sums of 60 terms: 1e-12 covers them."""
    N, T, B, D, beta, dt = 60, 4, 2, 0.9, 1.1, 1e-4
    L = inputs.box_side(N, 0.85)
    walk = np.cumsum(0.01 * inputs.rng(3).standard_normal((B, T + 1, 3, N)), axis=1)
    paths = inputs.fcc_lattice(N, L)[None, None] + walk
    out = []
    for s in (1.0, 2.0 ** k):
        prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L * s, rc=L / 2 * s, eps=s * s, sigma=s)], D, beta, dt,
                            "fp64")
        buf = prob.empty("cuda")
        prob.view(buf, 0).copy_(torch.from_numpy(paths * s))
        S, g = pamd.action_grad(prob, buf)
        torch.cuda.synchronize()
        out.append((S.cpu().numpy() / (s * s), prob.view(g, 0).cpu().numpy() / s))
    (S0, g0), (S1, g1) = out
    assert np.isfinite(g1).all() and np.abs(S1 - S0).max() <= 1e-12 * S0.max()
    assert np.abs(g1 - g0).max() <= 1e-12 * np.abs(g0).max()


@pytest.mark.parametrize("L", [16.0, 1024.0, 16384.0])
def test_pairs_at_the_cutoff(pamd, L):
    """Pairs a relative 1e-10 to 1e-6 inside and outside the cutoff, in boxes much larger than
    it and across their faces: the single-precision search may miss none, and the decision is
    that of the stored coordinates (their spacing moves a distance by 1e-11 at most).  A
    wrong decision would change the gradient by the pair's curvature, 1e-6 of it."""
    N, T, rc, D, beta, dt = 64, 6, 2.5, 0.9, 1.1, 1e-3
    rng = inputs.rng(int(L))
    grid = np.array([(x, y, z) for x in range(4) for y in range(4) for z in range(2)], float) * (L / 4)
    u = rng.standard_normal((32, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    paths = np.empty((1, T + 1, 3, N))
    for t in range(T + 1):
        off = rng.choice([-1, 1], 32) * 10.0 ** rng.uniform(-9.5 if L > 100 else -10, -6, 32)
        c = grid + 0.01 * rng.standard_normal((32, 3))
        paths[0, t, :, :32] = (c - 0.5 * rc * (1 + off)[:, None] * u).T
        paths[0, t, :, 32:] = (c + 0.5 * rc * (1 + off)[:, None] * u).T
    paths[0, :, :, ::5] += L * 3
    prob = pamd.Problem([pamd.System("lj", N, 3, T, 1, box=L, rc=rc)], D, beta, dt, "fp64")
    buf = prob.empty("cuda")
    prob.view(buf, 0).copy_(torch.from_numpy(paths))
    S, g = pamd.action_grad(prob, buf)
    torch.cuda.synchronize()
    So, go = oracle.action_grad(oracle.lennard_jones(L, rc), paths[0], D, beta, dt, nthreads=8)
    assert abs(S[0].item() - So) <= 1e-12 * So
    assert np.abs(prob.view(g, 0)[0].cpu().numpy() - go).max() <= 1e-12 * np.abs(go).max()
