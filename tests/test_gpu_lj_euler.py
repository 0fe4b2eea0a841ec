"""Euler-Maruyama paths of Lennard-Jones systems (lj_euler.cu) at the edges of their
launch shapes: one to eight CTAs per chain with uneven particle shares, one to 32 lanes
per particle, all pairs and Verlet lists (N around 192), lists that overflow, the largest
N.  Against the oracle fed the same normals; 12 steps keep the amplification of the
single-precision storage rounding (6e-8 of a coordinate) far below the tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import pamd_inputs as inputs  # noqa: E402


@pytest.fixture(scope="module")
def pamd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1907_09529_gb300 as m
    m.tune()
    return m


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("N,B,L,T", [(2, 1, 6.0, 12), (3, 200, 6.0, 3), (31, 3, 0, 12), (33, 1, 0, 12), (65, 160, 0, 3),
                                     (108, 4, 0, 12), (129, 2, 0, 12), (192, 1, 0, 12), (193, 1, 0, 12),
                                     (257, 80, 0, 3), (500, 2, 0, 12), (1024, 1, 0, 6), (250, 1, 40.0, 6),
                                     (40, 3, 0, 12), (49, 1, 0, 12), (50, 1, 0, 12), (57, 1, 0, 12),
                                     (64, 40, 0, 6)])
def test_paths_match_the_oracle(pamd, precision, N, B, L, T):
    D, beta, dt = 0.9, 1.1, 1e-4
    # the box of the whole FCC lattice that the particles occupy at density 0.85 (a partly
    # filled lattice in a smaller box overlaps, and the oracle's path explodes); L larger
    # than it: a droplet, denser than lists are sized for
    m = 1
    while 4 * m ** 3 < N:
        m += 1
    side = inputs.box_side(4 * m ** 3, 0.85)
    L = L or max(side, 3.2)
    rc = min(2.5, L / 2)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=rc)], D, beta, dt, precision)
    rng = inputs.rng(N)
    x0 = inputs.fcc_lattice(N, side if N > 4 else L) + 0.02 * rng.standard_normal((B, 3, N))
    z = rng.standard_normal((B, T + 1, 3, N))
    if precision == "fp32":
        x0, z = x0.astype(np.float32).astype(np.float64), z.astype(np.float32).astype(np.float64)
    buf, nbuf = prob.empty("cuda"), prob.empty("cuda")
    prob.view(buf, 0)[:, 0].copy_(torch.from_numpy(x0))
    prob.view(nbuf, 0).copy_(torch.from_numpy(z))
    pamd.euler_reference(prob, buf, noise=nbuf)
    torch.cuda.synchronize()
    want = oracle.euler_batch(oracle.lennard_jones(L, rc), x0, z[:, 1:], D, beta, dt, store_f32=precision == "fp32")
    got = prob.view(buf, 0).double().cpu().numpy()
    assert np.abs(got - want).max() <= (2e-5 if precision == "fp32" else 1e-11) * np.abs(want).max()


@pytest.mark.parametrize("N", [5, 108, 300])
def test_drawn_normals_equal_given_ones(pamd, N):
    """The normals drawn into the path give the path of the same normals passed in."""
    T, B, L = 7, 3, inputs.box_side(max(N, 64), 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=min(2.5, L / 2))], 1.0, 1.0, 1e-4)
    a, nbuf = prob.empty("cuda"), prob.empty("cuda")
    prob.view(a, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(N, L)))
    b = a.clone()
    for c in range(B):
        z = pamd.normals(11, 3, 0, c, (T + 1) * 3 * N)
        prob.view(nbuf, 0)[c].copy_(z.view(T + 1, 3, N))
    pamd.euler_reference(prob, a, seed=11, counter=3)
    pamd.euler_reference(prob, b, noise=nbuf)
    torch.cuda.synchronize()
    assert torch.equal(a, b)


@pytest.mark.parametrize("N", [57, 108, 200])
def test_long_paths_repeat(pamd, N):
    """Thousands of barrier phases, a cluster with an empty CTA among them: the same path
    in two calls, and no wait that ran out."""
    T, B, L = 3000, 5, inputs.box_side(256, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4)
    a = prob.empty("cuda")
    prob.view(a, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(256, L)[:, :N].copy()))
    b = a.clone()
    pamd.euler_reference(prob, a, seed=1, counter=2)
    pamd.euler_reference(prob, b, seed=1, counter=2)
    pamd.device_status()
    assert torch.equal(a, b) and bool(torch.isfinite(prob.view(a, 0)).all())


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("N,B", [(33, 1), (34, 19), (42, 2), (49, 3), (57, 1), (65, 9)])
def test_uneven_shares_repeat(pamd, precision, N, B):
    """Particle counts that eight CTAs cannot share equally, over thousands of barrier
    phases: the same path in two calls, and no wait that ran out."""
    T, L = 3000, inputs.box_side(256, 0.85)
    prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4, precision)
    a = prob.empty("cuda")
    prob.view(a, 0)[:, 0].copy_(torch.from_numpy(inputs.fcc_lattice(256, L)[:, :N].copy()))
    b = a.clone()
    pamd.euler_reference(prob, a, seed=1, counter=2)
    pamd.euler_reference(prob, b, seed=1, counter=2)
    pamd.device_status()
    assert torch.equal(a, b) and bool(torch.isfinite(prob.view(a, 0)).all())


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("N", [50, 64, 65, 108, 128, 129, 192, 193, 256, 300, 512, 513, 864, 1024])
def test_paths_do_not_depend_on_the_chains_beside_them(pamd, precision, N):
    """A chain's path is the same in calls of few chains (clusters of eight CTAs) and many
    (fewer CTAs a chain, one to four partial sums a lane), bit for bit."""
    T, L = 6, inputs.box_side(1372, 0.85)
    x0 = torch.from_numpy(inputs.fcc_lattice(1372, L)[:, :N].copy())
    paths = []
    for B in (1, 16, 30, 60, 100):
        prob = pamd.Problem([pamd.System("lj", N, 3, T, B, box=L, rc=2.5)], 1.0, 1.0, 1e-4, precision)
        buf = prob.empty("cuda")
        prob.view(buf, 0)[:, 0].copy_(x0)
        pamd.euler_reference(prob, buf, seed=1, counter=2)
        paths.append(prob.view(buf, 0)[:min(B, 16)].clone())
    pamd.device_status()
    for p in paths[2:]:
        assert torch.equal(p, paths[1])
    assert torch.equal(paths[0], paths[1][:1])
