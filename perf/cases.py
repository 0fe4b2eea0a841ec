"""The work a user of this package has it do, as measurable cases.

Every case is one call (or one short loop) of the package's public entry points on
paths of the kind the method meets: Euler-Maruyama / AR(1) oscillator paths, and
Lennard-Jones liquid paths that start on an FCC lattice and move by Brownian
dynamics.  A case is a dict of plain values:

  op         grad | action | update | euler | pamd | fragment
  kind       harmonic | lj
  precision  fp32 | fp64
  d          Cartesian dimensions
  shapes     systems "N:T:chains", comma separated (particles, steps, paths)
  dt         path discretisation step
  updates    (update) Metropolis-adjusted path updates per call
  events, n_sample, n_shift, l_min, l_max   (pamd) the path-accelerated MD loop
  steps, l_min, l_max                       (fragment) multilevel Monte Carlo steps

D = beta = k = 1, the Lennard-Jones liquid has reduced density 0.85, T* = 1 and the
cutoff min(2.5, L/2).
"""
import math

import torch

import paper_1907_09529_gb300 as pamd
from paper_1907_09529_gb300 import integrator

DENSITY = 0.85
ALIGN = 8          # a system starts at a multiple of 8 elements of the flat buffer
COARSE = 4         # steps between the points of a coarse Brownian-dynamics path


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # The 1D oscillator, one double-precision path of 1024 steps: the smallest call,
        # all latency and launches.
        {"name": "ho1d_grad_fp64", "op": "grad", "kind": "harmonic", "precision": "fp64", "d": 1,
         "shapes": "1:1024:1", "dt": 0.01},
        # The same path sampled: a hundred path updates in one call, replayed from a graph.
        {"name": "ho1d_update_fp64", "op": "update", "kind": "harmonic", "precision": "fp64", "d": 1,
         "shapes": "1:1024:1", "dt": 0.01, "updates": 100},
        # 64 long 3D oscillator paths: the memory-bound action and gradient ...
        {"name": "ho3d_grad", "op": "grad", "kind": "harmonic", "precision": "fp32", "d": 3,
         "shapes": "1:1048576:64", "dt": 0.005},
        # ... and one path update of all of them.
        {"name": "ho3d_update", "op": "update", "kind": "harmonic", "precision": "fp32", "d": 3,
         "shapes": "1:1048576:64", "dt": 0.005, "updates": 1},
        # One path of a small liquid: action and gradient for an outer sampler or optimiser.
        {"name": "lj108_grad", "op": "grad", "kind": "lj", "precision": "fp32", "d": 3,
         "shapes": "108:4096:1", "dt": 1e-4},
        # The action alone (monitoring, gradient-free moves).
        {"name": "lj500_action", "op": "action", "kind": "lj", "precision": "fp32", "d": 3,
         "shapes": "500:4096:2", "dt": 1e-4},
        # One path update of 8 long liquid paths: the largest ordinary job.
        {"name": "lj500_update", "op": "update", "kind": "lj", "precision": "fp32", "d": 3,
         "shapes": "500:16384:8", "dt": 1e-4, "updates": 1},
        # A batch of unlike liquids (odd sizes, 64 to 864 particles), two updates in one call.
        {"name": "ragged_update", "op": "update", "kind": "lj", "precision": "fp32", "d": 3,
         "shapes": "64:3001:1,97:4096:1,131:1024:1,187:2357:1,256:777:1,301:1500:1,367:2048:1,"
                   "411:903:1,500:1777:1,613:640:1,733:1111:1,864:2222:1", "dt": 1e-4, "updates": 2},
        # The plain double-precision form, for validation runs.
        {"name": "lj256_grad_fp64", "op": "grad", "kind": "lj", "precision": "fp64", "d": 3,
         "shapes": "256:512:2", "dt": 1e-4},
        # Start paths: sequential Euler-Maruyama of a few small liquids.
        {"name": "lj108_euler", "op": "euler", "kind": "lj", "precision": "fp32", "d": 3,
         "shapes": "108:1024:4", "dt": 1e-4},
        # The path-accelerated MD loop on 1D oscillator paths (N_path 4096, N_sample 1,
        # N_shift 64, levels 4..8; exact propagator, straight-line regrowth).
        {"name": "pamd_ho1d", "op": "pamd", "kind": "harmonic", "precision": "fp32", "d": 1,
         "shapes": "1:4096:8192", "dt": 0.4, "events": 4, "n_sample": 1, "n_shift": 64,
         "l_min": 4, "l_max": 8},
        # The multilevel sampler on 3D oscillator paths.
        {"name": "fragment_ho3d", "op": "fragment", "kind": "harmonic", "precision": "fp32", "d": 3,
         "shapes": "1:1024:4096", "dt": 0.05, "steps": 4, "l_min": 3, "l_max": 7},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fam = rng.choice(["ho_grad", "ho_update", "lj", "lj", "ragged", "lj64", "euler", "pamd", "fragment"])
    if fam in ("ho_grad", "ho_update"):
        N, d = rng.choice([1, 1, 1, 2, 5]), rng.choice([1, 2, 3])
        T = _log_int(rng, 64, 1 << 20)
        most = (1 << 26) * 3 // (N * d * (T + 1))
        fp64 = rng.random() < 0.4
        if fp64:
            most //= 8
        case = {"op": "grad", "kind": "harmonic", "precision": "fp64" if fp64 else "fp32", "d": d,
                "shapes": "%d:%d:%d" % (N, T, _log_int(rng, 1, max(1, min(4096 if fam == "ho_grad" else 64, most)))),
                "dt": 0.005}
        if fam == "ho_update":
            N, T, B = (int(v) for v in case["shapes"].split(":"))
            case.update(op="update", updates=rng.randint(1, 40) if N * d * T * B < 1 << 21 else 1)
        return case
    if fam in ("lj", "lj64"):
        N = _log_int(rng, 32, 864)
        units = _log_int(rng, 20000, 600000 if fam == "lj64" else 40000000)
        T = max(16, min(16384, _log_int(rng, 64, 16384), units // N))
        B = max(1, min(64, units // (N * T)))
        case = {"op": rng.choice(["grad", "action", "update"]), "kind": "lj",
                "precision": "fp64" if fam == "lj64" else "fp32", "d": 3,
                "shapes": "%d:%d:%d" % (N, T, B), "dt": 1e-4}
        if case["op"] == "update":
            case["updates"] = 1 if units > 2000000 or fam == "lj64" else rng.randint(1, 4)
        return case
    if fam == "ragged":
        shapes = ["%d:%d:%d" % (rng.randint(64, 864), _log_int(rng, 128, 4096), rng.choice([1, 1, 2]))
                  for _ in range(rng.randint(3, 10))]
        return {"op": "grad", "kind": "lj", "precision": "fp32", "d": 3, "shapes": ",".join(shapes),
                "dt": 1e-4}
    if fam == "euler":
        return {"op": "euler", "kind": "lj", "precision": rng.choice(["fp32", "fp32", "fp64"]), "d": 3,
                "shapes": "%d:%d:%d" % (_log_int(rng, 32, 512), _log_int(rng, 64, 512), rng.randint(1, 8)),
                "dt": 1e-4}
    T = _log_int(rng, 256, 8192)
    l_max = rng.randint(5, min(9, int(math.log2(T)) - 1))
    l_min = rng.randint(2, l_max)
    if fam == "pamd":
        return {"op": "pamd", "kind": "harmonic", "precision": "fp32", "d": 1,
                "shapes": "1:%d:%d" % (T, _log_int(rng, 64, (1 << 25) // T)), "dt": 0.4,
                "events": rng.randint(1, 4), "n_sample": rng.randint(1, 3),
                "n_shift": rng.randint(8, 128), "l_min": l_min, "l_max": l_max}
    d = rng.choice([2, 3])
    T = min(T, 4096)
    return {"op": "fragment", "kind": "harmonic", "precision": rng.choice(["fp32", "fp32", "fp64"]),
            "d": d, "shapes": "1:%d:%d" % (T, _log_int(rng, 64, (1 << 23) // T)), "dt": 0.05,
            "steps": rng.randint(1, 4), "l_min": l_min, "l_max": l_max}


def _shapes(case):
    return [tuple(int(v) for v in s.split(":")) for s in case["shapes"].split(",")]


def _box(N):
    L = (N / DENSITY) ** (1.0 / 3.0)
    return L, min(2.5, L / 2)


def _offsets(case):
    off, out = 0, []
    for N, T, B in _shapes(case):
        out.append(off)
        off = (off + B * (T + 1) * case["d"] * N + ALIGN - 1) // ALIGN * ALIGN
    return out, off


def _step(case):
    """Step size h of the path update: MALA's scaling with the dimension of a path."""
    dim = max(T * case["d"] * N for N, T, _ in _shapes(case))
    return 0.4 * case["dt"] * dim ** (-1.0 / 3.0)


# ---------------------------------------------------------------- inputs (from the seed alone)
def _lattice(N, L):
    """First N sites of an FCC lattice filling the box, [3][N]."""
    m = 1
    while 4 * m ** 3 < N:
        m += 1
    basis = [(0, 0, 0), (0.5, 0.5, 0), (0.5, 0, 0.5), (0, 0.5, 0.5)]
    sites = [(x + a + 0.25, y + b + 0.25, z + c + 0.25)
             for x in range(m) for y in range(m) for z in range(m) for a, b, c in basis][:N]
    return torch.tensor(sites, dtype=torch.float64).T.contiguous() * (L / m)


def _lj_dense_force(x, L, rc):
    """Forces of all pairs; x [B][3][N]."""
    src = rc ** -6
    duc = 4.0 * (-12.0 * src * src + 6.0 * src) / rc
    d = x[:, :, :, None] - x[:, :, None, :]
    d = d - L * torch.round(d / L)
    r2 = (d * d).sum(1)
    i2 = torch.where((r2 <= rc * rc) & (r2 > 0), 1.0 / r2, torch.zeros_like(r2))
    i6 = i2 * i2 * i2
    fs = 24.0 * i2 * i6 * (2.0 * i6 - 1.0) + duc * torch.sqrt(i2)
    return (fs[:, None] * d).sum(-1)


def _lj_path(N, T, B, dt, gen):
    """Brownian-dynamics liquid paths [B][T+1][3][N]: Euler-Maruyama with a coarse step
    from the FCC lattice, Brownian bridges between its points."""
    L, rc = _box(N)
    Tc = -(-T // COARSE)
    x = _lattice(N, L).to("cuda", torch.float32)[None].repeat(B, 1, 1)
    xi = torch.randn((Tc, B, 3, N), generator=gen, device="cuda") * math.sqrt(2 * dt * COARSE)
    pts = torch.empty((B, Tc + 1, 3, N), device="cuda")
    pts[:, 0] = x
    for t in range(Tc):
        # (a coarse step into a neighbour's core is kept short)
        x = x + (dt * COARSE * _lj_dense_force(x, L, rc)).clamp(-0.05, 0.05) + xi[t]
        pts[:, t + 1] = x
    out = torch.empty((B, Tc * COARSE + 1, 3, N), device="cuda")
    out[:, -1] = pts[:, -1]
    for b in range(B):
        w = torch.randn((Tc, COARSE, 3, N), generator=gen, device="cuda").mul_(math.sqrt(2 * dt)).cumsum(1)
        s = (torch.arange(1, COARSE + 1, device="cuda") / COARSE).view(1, -1, 1, 1)
        a, z = pts[b, :-1, None], pts[b, 1:, None]
        v = a + s * (z - a) + w - s * w[:, -1:]
        rows = out[b, :-1].view(Tc, COARSE, 3, N)
        rows[:, 0] = pts[b, :-1]
        rows[:, 1:] = v[:, :-1]
    return out[:, :T + 1]


def _ho_path(N, T, B, d, phi, var, gen):
    """Stationary AR(1) oscillator paths [B][T+1][d][N], x_{t+1} = phi x_t + s xi."""
    s, K = d * N, 1024
    nb = -(-(T + 1) // K)
    s_xi = math.sqrt(var * (1 - phi * phi))
    out = torch.empty((B, nb * K, s), device="cuda", dtype=torch.float32)
    p = phi ** torch.arange(K, device="cuda", dtype=torch.float64)
    for b0 in range(0, B, 64):
        b1 = min(B, b0 + 64)
        xi = torch.randn((b1 - b0, nb, K, s), generator=gen, device="cuda").double().mul_(s_xi)
        loc = (xi / p.view(1, 1, K, 1)).cumsum(2) * p.view(1, 1, K, 1)
        carry = torch.randn((b1 - b0, s), generator=gen, device="cuda").double() * math.sqrt(var)
        ends = []
        for k in range(nb):
            ends.append(carry)
            carry = loc[:, k, -1] + phi ** K * carry
        loc += torch.stack(ends, 1)[:, :, None] * (phi * p).view(1, 1, K, 1)
        out[b0:b1] = loc.view(b1 - b0, nb * K, s).float()
    return out[:, :T + 1].reshape(B, T + 1, d, N)


def _inputs(case, seed):
    """The flat path buffer in the layout of the package, in the case's precision."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    offs, span = _offsets(case)
    pos = torch.zeros(span, device="cuda", dtype=torch.float32 if case["precision"] == "fp32" else torch.float64)
    d, dt = case["d"], case["dt"]
    for (N, T, B), o in zip(_shapes(case), offs):
        v = pos[o:o + B * (T + 1) * d * N].view(B, T + 1, d, N)
        if case["op"] == "euler":
            x0 = _lattice(N, _box(N)[0]).to("cuda")
            v[:, 0] = x0 + 0.03 * torch.randn((B, 3, N), generator=gen, device="cuda")
        elif case["kind"] == "lj":
            v.copy_(_lj_path(N, T, B, dt, gen))
        elif case["op"] == "pamd":
            v.copy_(_ho_path(N, T, B, d, math.exp(-dt), 1.0, gen))
        else:
            v.copy_(_ho_path(N, T, B, d, 1 - dt, 2 * dt / (1 - (1 - dt) ** 2), gen))
    return pos


def prepare(case, seed):
    pos = _inputs(case, seed)
    systems = []
    for N, T, B in _shapes(case):
        if case["kind"] == "lj":
            L, rc = _box(N)
            systems.append(pamd.System("lj", N, 3, T, B, box=L, rc=rc))
        else:
            systems.append(pamd.System("harmonic", N, case["d"], T, B, k=1.0))
    p = pamd.Problem(systems, 1.0, 1.0, case["dt"], case["precision"],
                     ho_exact_propagator=case["op"] == "pamd", regenerate_flat=case["op"] == "pamd")
    st = {"op": case["op"], "p": p, "pos": pos, "seed": seed, "counter": 0, "case": case}
    if case["op"] in ("grad", "action"):
        st["S"] = torch.empty(p.n_chains, dtype=torch.float64, device="cuda")
        st["grad"] = torch.zeros_like(pos)
    elif case["op"] == "update":
        st["S"], st["grad"] = pamd.action_grad(p, pos)
        st["nacc"] = torch.zeros(p.n_chains, dtype=torch.int32, device="cuda")
        st["h"] = _step(case)
    elif case["op"] == "pamd":
        st["loop"] = integrator.PamdIntegrator(p, case["n_shift"], case["n_sample"], case["l_min"],
                                               case["l_max"], seed=seed)
    elif case["op"] == "fragment":
        st["nacc"] = torch.zeros(p.n_chains, dtype=torch.int32, device="cuda")
        st["nprop"] = torch.zeros(p.n_chains, dtype=torch.int32, device="cuda")
    return st


def run(state):
    op, p, case = state["op"], state["p"], state["case"]
    if op == "grad":
        pamd.action_grad(p, state["pos"], state["S"], state["grad"])
        return state["S"], state["grad"]
    if op == "action":
        pamd.action(p, state["pos"], state["S"])
        return (state["S"],)
    if op == "update":
        n = case["updates"]
        pamd.path_update(p, state["pos"], state["grad"], state["S"], state["h"], n, seed=state["seed"],
                         counter=state["counter"], n_accepted=state["nacc"])
        state["counter"] += n
        return state["pos"], state["grad"], state["S"], state["nacc"]
    if op == "euler":
        pamd.euler_reference(p, state["pos"], seed=state["seed"], counter=state["counter"])
        state["counter"] += 1
        return (state["pos"],)
    if op == "pamd":
        traj = state["loop"].run(state["pos"], case["events"])
        return traj, state["pos"], state["loop"].n_accepted, state["loop"].n_proposed
    n = case["steps"]
    pamd.fragment_mc(p, state["pos"], case["l_min"], case["l_max"], n, seed=state["seed"],
                     counter=state["counter"], n_accepted=state["nacc"], n_proposed=state["nprop"])
    state["counter"] += n
    return state["pos"], state["nacc"], state["nprop"]


def work(case):
    """Bytes: every input read once and every output written once.  Flops (FMA = 2): 75 per
    unordered Lennard-Jones pair within the cutoff with the gradient, 44 without, and 23
    per particle-step; 10 per oscillator coordinate; 12 per proposed coordinate of an update
    (its random numbers not counted)."""
    e = 4 if case["precision"] == "fp32" else 8
    d, op = case["d"], case["op"]
    elems = sum(B * (T + 1) * d * N for N, T, B in _shapes(case))
    flops = 0.0
    for N, T, B in _shapes(case):
        if case["kind"] == "lj":
            pairs = 0.5 * N * min(N - 1, 4.0 / 3.0 * math.pi * _box(N)[1] ** 3 * DENSITY)
            flops += B * T * (pairs * (44 if op in ("action", "euler") else 75) + 23 * N)
        else:
            flops += 10.0 * B * T * d * N
    if op == "action":
        return {"bytes": elems * e, "flops": flops}
    if op == "grad":
        return {"bytes": 2 * elems * e, "flops": flops}
    if op == "update":
        return {"bytes": 4 * elems * e, "flops": case["updates"] * (flops + 12 * elems)}
    if op == "euler":
        return {"bytes": elems * e, "flops": flops}
    if op == "pamd":
        return {"bytes": 2 * elems * e, "flops": case["events"] * case["n_sample"] * 2 * flops}
    return {"bytes": 2 * elems * e, "flops": case["steps"] * 2 * flops}


# ---------------------------------------------------------------- the same in 64 bits, plain torch
M32 = 0xFFFFFFFF


def _mul32(c, v):
    """High and low words of the product of the constant c and v (32-bit values in int64)."""
    return (c * (v >> 16) + ((c * (v & 0xFFFF)) >> 16)) >> 16, (c * v) & M32


def _philox(x, y, z, w, seed):
    """Philox4x32-10; counter words as int64 tensors or numbers."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, x)
        h1, l1 = _mul32(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x, y, z, w


def _words(stream, counter, chain, first, seed):
    """The four words of counter (first, chain, counter, stream); first, chain int64 tensors."""
    zero = torch.zeros_like(first + chain)
    hi = ((counter >> 32) & 0xFFFF) | (stream << 16)
    return _philox(first + zero, chain + zero, zero + (counter & M32), zero + hi, seed)


def _normals(stream, counter, chain, n, seed):
    """Normals of elements 0..n-1 of one chain (Box-Muller of 24-bit uniforms)."""
    g = torch.arange((n + 3) // 4, device="cuda", dtype=torch.int64)
    w = _words(stream, counter, torch.tensor(chain, device="cuda"), g, seed)
    out = torch.empty((g.numel(), 4), device="cuda", dtype=torch.float64)
    for q in (0, 2):
        r = torch.sqrt(-2 * torch.log(((w[q] >> 8) + 1).double() / 2 ** 24))
        a = 2 * math.pi * (w[q + 1] >> 8).double() / 2 ** 24
        out[:, q], out[:, q + 1] = r * torch.cos(a), r * torch.sin(a)
    return out.view(-1)[:n]


def _uniform53(w):
    return (((w[0] >> 5) * 67108864 + (w[1] >> 6)).double() + 1.0) / 2.0 ** 53


class _Pairs:
    """Pairs i < j of consecutive slices X [S][3][N] that can be within the cutoff at any of them."""

    def __init__(self, X, L, rc):
        c = X[X.shape[0] // 2]
        m = (X - c).norm(dim=1).amax(0)
        d = c[:, :, None] - c[:, None, :]
        d = d - L * torch.round(d / L)
        near = d.norm(dim=0) <= rc + m[:, None] + m[None, :] + 1e-9
        self.i, self.j = torch.nonzero(torch.triu(near, 1), as_tuple=True)
        d = X[:, :, self.i] - X[:, :, self.j]
        self.d = d - L * torch.round(d / L)
        r2 = (self.d * self.d).sum(1)
        i2 = torch.where(r2 <= rc * rc, 1.0 / r2, torch.zeros_like(r2))
        i6 = i2 * i2 * i2
        src = rc ** -6
        self.fs = 24.0 * i2 * i6 * (2.0 * i6 - 1.0) + 4.0 * (-12.0 * src * src + 6.0 * src) / rc * torch.sqrt(i2)
        self.bc = (24.0 * i2 * i6 * (26.0 * i6 - 7.0) + self.fs) * i2
        self.like = X

    def _sum(self, v):
        out = torch.zeros_like(self.like)
        return out.index_add_(2, self.i, v).index_add_(2, self.j, -v)

    def force(self):
        return self._sum(self.fs[:, None] * self.d)

    def hvp(self, V):
        v = V[:, :, self.i] - V[:, :, self.j]
        dv = (self.d * v).sum(1)
        return self._sum((self.bc * dv)[:, None] * self.d - self.fs[:, None] * v)


def _action_grad64(case, shape, x):
    """S and gradient of one path x [T+1][d][N]."""
    a = case["dt"]
    ginv = 1.0 / (2.0 * case["dt"])
    if case["kind"] == "harmonic":
        r = x[1:] - x[:-1] + a * x[:-1]
        g = torch.zeros_like(x)
        g[1:] = r
        g[:-1] += (a - 1.0) * r
        return (r * r).sum() * 0.5 * ginv, g.mul_(ginv)
    N, T, _ = shape
    L, rc = _box(N)
    g = torch.empty_like(x)
    S = torch.zeros((), device="cuda", dtype=torch.float64)
    last = torch.zeros_like(x[0])
    for t0 in range(0, T, 64):
        t1 = min(T, t0 + 64)
        P = _Pairs(x[t0:t1], L, rc)
        r = x[t0 + 1:t1 + 1] - x[t0:t1] - a * P.force()
        S += (r * r).sum() * 0.5 * ginv
        g[t0:t1] = (torch.cat([last[None], r[:-1]]) - r + a * P.hvp(r)) * ginv
        last = r[-1]
    g[T] = last * ginv
    return S, g


def _paths(case, pos):
    """(chain, shape, view of the path) of every chain."""
    offs, _ = _offsets(case)
    c = 0
    for shape, o in zip(_shapes(case), offs):
        N, T, B = shape
        v = pos[o:o + B * (T + 1) * case["d"] * N].view(B, T + 1, case["d"], N)
        for b in range(B):
            yield c, shape, v[b]
            c += 1


def _exact_update(case, seed, pos, grad, S):
    h = _step(case)
    for c, shape, x in _paths(case, pos):
        g = [v for q, _, v in _paths(case, grad) if q == c][0]
        s0, g0 = _action_grad64(case, shape, x)
        for u in range(case["updates"]):
            z = _normals(1, u, c, x.numel(), seed).view_as(x)
            y = x - h * g0 + math.sqrt(2 * h) * z
            y[0] = x[0]
            s1, g1 = _action_grad64(case, shape, y)
            qf = ((y - x + h * g0)[1:] ** 2).sum()
            qr = ((x - y + h * g1)[1:] ** 2).sum()
            la = (s0 - s1) - qr / (4 * h) + qf / (4 * h)
            first = torch.zeros((), device="cuda", dtype=torch.int64)
            w = _words(2, u, torch.tensor(c, device="cuda"), first, seed)
            if bool(torch.log(_uniform53(w)) < la):
                x.copy_(y)
                s0, g0 = s1, g1
        g.copy_(g0)
        S[c] = s0


def _exact_fragment(case, shape, x, seed, counter, drift, cS):
    """One multilevel Monte Carlo step of all chains; x [B][T+1][M], updated in place."""
    N, T, B = shape
    M, dt = case["d"] * N, case["dt"]
    sig, c0 = math.sqrt(2 * dt), 1.0 / (4 * dt)
    chain = torch.arange(B, device="cuda", dtype=torch.int64)
    w = _words(3, counter, chain, torch.zeros_like(chain), seed)
    l = case["l_min"] + w[0] % (case["l_max"] - case["l_min"] + 1)
    o = w[1] % (1 << l)
    first = torch.where(o > 0, o, 1 << l)[:, None]
    l = l[:, None]
    nfrag = 1 + torch.where(first < T, ((T - 1 - first) >> l) + 1, 0)
    t = torch.arange(1, T + 1, device="cuda")[None]
    f = torch.where(t - 1 < first, 0, 1 + ((t - 1 - first) >> l))
    fa = torch.where(f == 0, 0, first + ((f - 1) << l))
    nose = f == nfrag - 1
    fb = torch.where(nose, T, first + (f << l))
    e = torch.arange((T + 1) * M, device="cuda", dtype=torch.int64)
    z = torch.empty((B, T + 1, M), device="cuda", dtype=torch.float64)
    for b0 in range(0, B, 1024):  # normals of a batch of chains at once
        cb = chain[b0:b0 + 1024, None]
        g = torch.arange(((T + 1) * M + 3) // 4, device="cuda", dtype=torch.int64)[None]
        v = _words(4, counter, cb, g, seed)
        q = []
        for k in (0, 2):
            r = torch.sqrt(-2 * torch.log(((v[k] >> 8) + 1).double() / 2 ** 24))
            a = 2 * math.pi * (v[k + 1] >> 8).double() / 2 ** 24
            q += [r * torch.cos(a), r * torch.sin(a)]
        z[b0:b0 + 1024] = torch.stack(q, -1).view(cb.shape[0], -1)[:, e].view(-1, T + 1, M)
    z[:, 0] = 0
    C = (sig * z).cumsum(1)

    def at(v, idx):
        return torch.gather(v, 1, idx[..., None].expand(-1, -1, M))

    W = C[:, 1:] - at(C, fa)
    Wb = at(C, fb) - at(C, fa)
    xa, xb = at(x, fa), at(x, fb)
    s = ((t - fa).double() / (fb - fa).double())[..., None]
    y = torch.where(nose[..., None], xa + W, xa + s * (xb - xa) + W - s * Wb)
    y = torch.where(((t == fb) & ~nose)[..., None], x[:, 1:], y)
    y0 = torch.cat([x[:, :1], y[:, :-1]], 1)
    y0 = torch.where((t - 1 == fa)[..., None], x[:, :-1], y0)
    x0, x1 = x[:, :-1], x[:, 1:]
    r, rt = x1 - x0 + drift * x0, y - y0 + drift * y0
    dS = ((rt - r) * (rt + r)).sum(-1)
    dS0 = ((y - y0 - x1 + x0) * (y - y0 + x1 - x0)).sum(-1)
    F = int(nfrag.max())
    sums = [torch.zeros((B, F), device="cuda", dtype=torch.float64).scatter_add_(1, f, v) for v in (dS, dS0)]
    u = _uniform53(_words(5, counter, chain[:, None], torch.arange(F, device="cuda", dtype=torch.int64)[None], seed))
    acc = torch.gather(torch.log(u) < sums[1] * c0 - sums[0] * cS, 1, f)
    move = acc & (nose | ((fb - fa >= 2) & (t < fb)))
    x[:, 1:] = torch.where(move[..., None], y, x1)


def exact(case, seed):
    pos = _inputs(case, seed).double()
    op, shapes = case["op"], _shapes(case)
    n = sum(B for _, _, B in shapes)
    if op in ("grad", "action", "update"):
        S = torch.zeros(n, device="cuda", dtype=torch.float64)
        grad = torch.zeros_like(pos)
        if op == "update":
            _exact_update(case, seed, pos, grad, S)
            return pos, grad, S, None
        for (c, shape, x), (_, _, g) in zip(_paths(case, pos), _paths(case, grad)):
            S[c], g0 = _action_grad64(case, shape, x)
            g.copy_(g0)
        return (S, grad) if op == "grad" else (S,)
    if op == "euler":
        sig = math.sqrt(2 * case["dt"])
        offs, _ = _offsets(case)
        c = 0
        for (N, T, B), o in zip(shapes, offs):
            L, rc = _box(N)
            v = pos[o:o + B * (T + 1) * 3 * N].view(B, T + 1, 3, N)
            z = torch.stack([_normals(0, 0, c + b, (T + 1) * 3 * N, seed).view(T + 1, 3, N) for b in range(B)])
            for t in range(T):
                v[:, t + 1] = v[:, t] + case["dt"] * _lj_dense_force(v[:, t], L, rc) + sig * z[:, t + 1]
            c += B
        return (pos,)
    N, T, B = shapes[0]
    x = pos[:B * (T + 1) * case["d"] * N].view(B, T + 1, case["d"] * N)
    dt = case["dt"]
    if op == "fragment":
        for u in range(case["steps"]):
            _exact_fragment(case, shapes[0], x, seed, u, dt, 1.0 / (4 * dt))
        return pos, None, None
    phi = math.exp(-dt)
    ns, traj = case["n_shift"], []
    for ev in range(case["events"]):
        for u in range(case["n_sample"]):
            _exact_fragment(case, shapes[0], x, seed, ev * case["n_sample"] + u, 1 - phi,
                            1.0 / (2 * (1 - phi * phi)))
        traj.append(x[:, 1:ns + 1].reshape(-1).clone())
        x.copy_(torch.cat([x[:, ns:], x[:, -1:].expand(-1, ns, -1)], 1).clone())
    return torch.stack(traj), pos, None, None
