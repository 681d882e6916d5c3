"""The work that users of the library have it do, as cases that can be timed and compared.

A case is one pass through the public entry points (`Context`, `MLP`, `Lift`, `moments_rot`); its sizes are
those of this repository's tests and benchmark workloads or odd ones of the same ranges.  Shapes are unions of
balls drawn from a seed: knots uniform in ellipsoids (A) or in a solid torus (B), radii from a few levels.
`exact` computes the same results in 64 bits with plain torch: direct nonequispaced sums, no spreading.
"""
import math

import numpy as np
import torch

import paper_1711_05075_gb300 as bc

P = 2.0  # translation period
LIFT_L, LIFT_PR = 0.1, 0.4  # cone height and lifted period of the lifted workload
LEVELS = {1: (0.05,), 2: (0.04, 0.08), 3: (0.02, 0.04, 0.08), 4: (0.01, 0.02, 0.04, 0.08),
          8: (0.01, 0.015, 0.02, 0.03, 0.04, 0.05, 0.06, 0.08)}
PROBS = {1: (1.0,), 2: (0.5, 0.5), 3: (0.5, 0.3, 0.2), 4: (0.4, 0.3, 0.2, 0.1), 8: (0.125,) * 8}


def listed():
    return [
        # the smallest call: 128-ball ellipsoid and torus on a 32^3 grid, identity rotation; latency and launches
        {"name": "pair_32", "kind": "pair", "N": 32, "W": 6, "L": 2, "nA": 128, "nB": 128, "k": 1, "precision": 0},
        # shape complementarity of a mid-sized pair under a few rotations, odd counts
        {"name": "score_64", "kind": "score", "N": 64, "W": 8, "L": 4, "nA": 2311, "nB": 741, "k": 5},
        # the benchmark's headline: one correlation of two 20,000-ball shapes on the 128^3 grid
        {"name": "pair_128", "kind": "pair", "N": 128, "W": 8, "L": 4, "nA": 20000, "nB": 20000, "k": 1,
         "precision": 0},
        # the largest grid: the same pair at 256^3
        {"name": "pair_256", "kind": "pair", "N": 256, "W": 8, "L": 4, "nA": 20000, "nB": 20000, "k": 1,
         "precision": 0},
        # the split-precision option of the same correlation
        {"name": "split_128", "kind": "pair", "N": 128, "W": 8, "L": 4, "nA": 20000, "nB": 20000, "k": 1,
         "precision": 1},
        # docking sweep: peaks of one receptor with a ligand under many rotations
        {"name": "sweep_96", "kind": "sweep", "N": 96, "W": 8, "L": 4, "nA": 50000, "nB": 5000, "k": 200},
        # a ragged batch of new pairs: uploaded from page-locked host memory, one peak per pair
        {"name": "ragged_96", "kind": "ragged", "N": 96, "W": 8, "L": 4, "pairs": 24, "lo": 1000, "hi": 100000},
        # time-critical queries at arbitrary translations from the lowest modes of one configuration
        {"name": "query_128", "kind": "query", "N": 128, "W": 8, "L": 4, "nA": 20000, "nB": 20000, "modes": 4096,
         "pts": 4096},
        # nonequiradius (4D lifted) correlation, the section r = 0
        {"name": "lifted_128", "kind": "lifted", "N": 128, "Nr": 32, "nA": 5000, "nB": 5000, "sections": 1},
        # Fourier moments of a ligand under many rotations (features of the learned proposal)
        {"name": "moments_4096", "kind": "moments", "N": 96, "W": 8, "L": 4, "nA": 5000, "k": 4096},
        # ranking rotations: the network's forward pass over a full rotation set
        {"name": "predict_16384", "kind": "mlp", "H": 256, "n": 16384, "train": False},
        # one training batch: forward, loss and every gradient
        {"name": "grads_8192", "kind": "mlp", "H": 256, "n": 8192, "train": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "score", "sweep", "ragged", "query", "lifted", "moments", "mlp"])
    N = rng.choice([32, 64, 96, 128])
    W = rng.choice([6, 8, 8, 8, 9, 10])
    L = rng.choice([1, 2, 3, 4, 4, 4, 8])
    if kind == "pair":
        N = rng.choice([32, 64, 96, 128, 256])
        return {"kind": "pair", "N": N, "W": W, "L": min(L, 4) if N == 256 else L, "nA": _log(rng, 1, 100000),
                "nB": _log(rng, 1, 100000), "k": 1 if N == 256 else rng.choice([1, 1, 2, 3, 7]),
                "precision": rng.choice([0, 0, 0, 0, 1])}
    if kind == "score":
        return {"kind": "score", "N": N, "W": W, "L": L, "nA": _log(rng, 50, 50000), "nB": _log(rng, 50, 50000),
                "k": rng.choice([1, 2, 3, 7])}
    if kind == "sweep":
        N = rng.choice([32, 64, 96])
        return {"kind": "sweep", "N": N, "W": W, "L": 4 if L == 8 else L, "nA": _log(rng, 500, 50000),
                "nB": _log(rng, 100, 5000), "k": _log(rng, 10, 200)}
    if kind == "ragged":
        N = rng.choice([32, 64, 96])
        hi = _log(rng, 3000, 100000)
        return {"kind": "ragged", "N": N, "W": W, "L": 4 if L == 8 else L, "pairs": _log(rng, 2, 24),
                "lo": _log(rng, 100, 2000), "hi": hi}
    if kind == "query":
        return {"kind": "query", "N": N, "W": W, "L": L, "nA": _log(rng, 100, 20000), "nB": _log(rng, 100, 20000),
                "modes": _log(rng, 64, 8192), "pts": _log(rng, 1, 20000)}
    if kind == "lifted":
        return {"kind": "lifted", "N": N, "Nr": rng.choice([16, 32, 32, 64]), "nA": _log(rng, 30, 10000),
                "nB": _log(rng, 30, 10000), "sections": rng.choice([1, 1, 2, 3])}
    if kind == "moments":
        return {"kind": "moments", "N": N, "W": W, "L": L, "nA": _log(rng, 100, 20000), "k": _log(rng, 64, 4096)}
    return {"kind": "mlp", "H": rng.choice([64, 128, 256, 256, 512]), "n": _log(rng, 64, 8192),
            "train": rng.choice([True, False])}


# ---------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + stream)
    return g


def _u(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32)


def _ball_points(g, n):
    d = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float32)
    return d / d.norm(dim=1, keepdim=True).clamp_min(1e-12) * _u(g, n, 1) ** (1.0 / 3.0)


def _ellipsoid(g, n):
    return _ball_points(g, n) * torch.tensor([0.5, 0.35, 0.25], device="cuda")


def _union(g, n):
    """Knots of three ellipsoids of random centre and semi-axes (a receptor)."""
    c, a = _u(g, 3, 3) * 0.6 - 0.3, _u(g, 3, 3) * 0.2 + 0.15
    which = torch.randint(0, 3, (n,), generator=g, device="cuda")
    return c[which] + a[which] * _ball_points(g, n)


def _torus(g, n):
    t, f, s = 2 * math.pi * _u(g, n), 2 * math.pi * _u(g, n), 0.12 * _u(g, n).sqrt()
    rho = 0.4 + s * f.cos()
    return torch.stack([rho * t.cos(), rho * t.sin(), s * f.sin()], dim=1)


def _levels(g, n, L):
    cdf = torch.tensor(PROBS[L], device="cuda").cumsum(0)
    return torch.searchsorted(cdf, _u(g, n), right=True).clamp_max(L - 1).to(torch.int32)


def _quats(seed, k):
    """k uniform random rotations (host, float32)."""
    r = np.random.RandomState(seed % (1 << 31))
    q = r.standard_normal((k, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    q[q[:, 0] < 0] *= -1.0
    return q.astype(np.float32)


def _two_shapes(case, seed):
    """((xyz A, levels A), (xyz B, levels B)) on the GPU."""
    ga, gb = _gen(seed, 1), _gen(seed, 2)
    A = _union(ga, case["nA"]) if case["kind"] == "sweep" else _ellipsoid(ga, case["nA"])
    return (A, _levels(ga, case["nA"], case["L"])), (_torus(gb, case["nB"]),
                                                     _levels(gb, case["nB"], case["L"]))


def _pair_quats(case, seed):
    return np.array([[1, 0, 0, 0]], np.float32) if case.get("k", 1) == 1 else _quats(seed, case["k"])


def _ragged_shapes(case, seed):
    """Page-locked host arrays [(xyz, level)] of 2 x pairs shapes, A and B in turn."""
    r = np.random.RandomState(seed % (1 << 31))
    lo, hi = min(case["lo"], case["hi"]), max(case["lo"], case["hi"])
    out = []
    for i in range(2 * case["pairs"]):
        n = int(round(math.exp(r.uniform(math.log(lo), math.log(hi)))))
        g = _gen(seed, 100 + i)
        x = _torus(g, n) if i & 1 else _union(g, n)
        out.append((x.cpu().pin_memory(), _levels(g, n, case["L"]).cpu().pin_memory()))
    return out


def _lift_knots(seed, n, stream):
    g = _gen(seed, stream)
    x = _torus(g, n) if stream & 1 else _ellipsoid(g, n)
    return torch.cat([x, 0.01 + 0.08 * _u(g, n, 1)], dim=1).contiguous()


def _lift_sections(case):
    return (0.0, 0.02, -0.03)[: case["sections"]]


def _mlp_inputs(case, seed):
    """(initial parameters, feature rows X (n x 144), targets)."""
    H, n, g = case["H"], case["n"], _gen(seed, 3)

    def he(fan, count):
        return (_u(g, count) * 2 - 1) * math.sqrt(6.0 / fan)
    zero = torch.zeros(H, device="cuda")
    params = torch.cat([he(132, H * 132), zero, he(H, H * H), zero, he(H, H), zero[:1]])
    q = torch.randn((n, 4), generator=g, device="cuda")
    q = q / q.norm(dim=1, keepdim=True) * torch.where(q[:, :1] < 0, -1.0, 1.0)
    # the receptor's moments are the same in every row, the ligand's vary with the rotation
    X = torch.cat([q, (_u(g, 1, 64) ** 2).expand(n, 64), _u(g, n, 64) ** 2,
                   torch.zeros((n, 12), device="cuda")], dim=1).contiguous()
    return params, X, torch.randn(n, generator=g, device="cuda")


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "mlp":
        # the network lives on a context's device and stream
        s["ctx"] = bc.Context(32, 6, LEVELS[2], P)
        params, s["X"], s["t"] = _mlp_inputs(case, seed)
        s["net"] = bc.MLP(s["ctx"], case["H"], params.cpu().numpy())
        s["train"] = case["train"]
        return s
    if kind == "lifted":
        s["lift"] = bc.Lift(case["N"], case["Nr"], LIFT_L, P, LIFT_PR)
        s["A"], s["B"] = _lift_knots(seed, case["nA"], 4), _lift_knots(seed, case["nB"], 5)
        s["q"], s["sections"] = _quats(seed, 1)[0], _lift_sections(case)
        return s
    s["ctx"] = ctx = bc.Context(case["N"], case["W"], LEVELS[case["L"]], P, precision=case.get("precision", 0))
    if kind == "ragged":
        s["shapes"], s["q"] = _ragged_shapes(case, seed), _quats(seed, case["pairs"])
        return s
    if kind == "moments":
        g = _gen(seed, 2)
        s["B"] = ctx.shape(_torus(g, case["nA"]), _levels(g, case["nA"], case["L"]))
        s["q"] = torch.from_numpy(_quats(seed, case["k"])).cuda()
        return s
    a, b = _two_shapes(case, seed)
    s["A"], s["B"] = ctx.shape(*a), ctx.shape(*b)
    if kind == "query":
        s["query"] = ctx.query(s["A"], s["B"], _quats(seed, 1)[0], min(case["modes"], ((case["N"] - 1) ** 3 + 1) // 2))
        s["t"] = _u(_gen(seed, 6), case["pts"], 3) * P - P / 2
    else:
        s["q"] = _pair_quats(case, seed)
    return s


def run(s):
    kind = s["kind"]
    if kind == "pair":
        return s["ctx"].correlate(s["A"], s["B"], s["q"])
    if kind == "score":
        return s["ctx"].score(s["A"], s["B"], s["q"], 0.02, 2.0)
    if kind == "sweep":
        return s["ctx"].sweep(s["A"], s["B"], s["q"])
    if kind == "ragged":
        shapes = s["ctx"].shapes(s["shapes"])
        _, peak, arg = s["ctx"].pairs(shapes[0::2], shapes[1::2], s["q"])
        for x in shapes:
            x.close()
        return peak, arg
    if kind == "query":
        return s["query"].eval(s["t"])
    if kind == "lifted":
        return s["lift"].correlate(s["A"], s["B"], s["q"], s["sections"])
    if kind == "moments":
        return bc.moments_rot(s["ctx"], s["B"], s["q"])
    return s["net"].grads(s["X"], s["t"]) if s["train"] else s["net"].predict(s["X"])


# ---------------------------------------------------------------- what a pass cannot do without
def _fft_flops(points):
    return 5.0 * points * math.log2(points)


def work(case):
    kind = case["kind"]
    if kind == "mlp":
        # every weight once per row forward, twice more backward (the first layer has no input gradient)
        H, n, m = case["H"], case["n"], 132 * case["H"] + case["H"] ** 2 + 2 * case["H"] + case["H"] + 1
        fwd = 2.0 * n * (132 * H + H * H + H)
        back = 2.0 * n * (132 * H + 2 * H * H + 2 * H)
        by = 4.0 * (n * 132 + n + m + (m + n if case["train"] else 0))
        return {"bytes": by, "flops": fwd + (back if case["train"] else 0)}
    N = case["N"]
    if kind == "lifted":
        n, modes = case["nA"] + case["nB"], N ** 3 * case["Nr"] // 2
        return {"bytes": 16.0 * n + 4.0 * N ** 3 * case["sections"],
                "flops": 2.0 * 8 ** 4 * n + 2 * _fft_flops(modes) + case["sections"] * (8.0 * modes + _fft_flops(N ** 3) / 2)}
    if kind == "query":
        m = min(case["modes"], ((N - 1) ** 3 + 1) // 2)
        return {"bytes": 24.0 * m + 16.0 * case["pts"], "flops": 8.0 * m * case["pts"]}
    if kind == "moments":
        return {"bytes": 16.0 * case["nA"] + (16 + 4 * 64) * case["k"], "flops": 12.0 * 64 * case["nA"] * case["k"]}
    # a shape's spectrum: W^3 stencil cells per knot, a transform keeping N^3 / 2 modes per level, the level sum
    spectrum = case["L"] * (_fft_flops(N ** 3 / 2) + 2.0 * N ** 3)
    if kind == "ragged":
        lo, hi = min(case["lo"], case["hi"]), max(case["lo"], case["hi"])
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        nk, ns, k, out = 2 * case["pairs"] * mean, 2 * case["pairs"], case["pairs"], 8.0 * case["pairs"]
    else:
        k = case["k"]
        nk, ns = case["nA"] + k * case["nB"], 1 + k
        out = 8.0 * k if kind == "sweep" else 4.0 * N ** 3 * k
    knots = nk if kind == "ragged" else case["nA"] + case["nB"]
    return {"bytes": 16.0 * knots + out,
            "flops": 2.0 * case["W"] ** 3 * nk + ns * spectrum + k * (_fft_flops(N ** 3) / 2 + 3.0 * N ** 3)}


# ---------------------------------------------------------------- the same results in 64 bits
def _rotation(q):
    w, x, y, z = (float(v) for v in np.asarray(q, np.float64) / np.linalg.norm(np.asarray(q, np.float64)))
    return torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                         [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                         [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]],
                        dtype=torch.float64, device="cuda")


def _fft_modes(N):
    return torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda").round()


def _phases(x, m, period=P):
    """exp(-2 pi i m x / period), (len(m), len(x))."""
    a = (m[:, None] * x[None, :] / period)
    a = -2 * math.pi * (a - a.round())
    return torch.complex(a.cos(), a.sin())


def _ball_ft(r, k):
    """4 pi (sin kr - kr cos kr) / k^3, the transform of a ball's indicator (series near kr = 0)."""
    x = k * r
    x2 = x * x
    series = 1 / 3 - x2 / 30 + x2 ** 2 / 840 - x2 ** 3 / 45360 + x2 ** 4 / 3991680 - x2 ** 5 / 518918400
    xs = torch.where(x < 0.3, torch.ones_like(x), x)
    return 4 * math.pi * r ** 3 * torch.where(x < 0.3, series, (xs.sin() - xs * xs.cos()) / xs ** 3)


def _ndft(x, mx, my, mz):
    """sum_j exp(-2 pi i m . x_j / P) on mx x my x mz, by direct sums."""
    out = torch.zeros((len(mx) * len(my), len(mz)), dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 25) // (len(mx) * len(my)))
    for i in range(0, x.shape[0], step):
        c = x[i:i + step]
        xy = (_phases(c[:, 0], mx)[:, None, :] * _phases(c[:, 1], my)[None, :, :]).reshape(-1, c.shape[0])
        out += xy @ _phases(c[:, 2], mz).T
    return out.reshape(len(mx), len(my), len(mz))


def _spectrum(x, level, N, weights):
    """sum_l weights[l](k) S_l(m) for m_z in [0, N/2); modes with a component -N/2 are zero."""
    m, mz = _fft_modes(N), torch.arange(N // 2, dtype=torch.float64, device="cuda")
    k = 2 * math.pi / P * (m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2).sqrt()
    F = torch.zeros((N, N, N // 2), dtype=torch.complex128, device="cuda")
    for l, w in enumerate(weights):
        F += w(k) * _ndft(x[level == l], m, m, mz)
    F[N // 2] = 0
    F[:, N // 2] = 0
    return F


def _weights(case):
    if case["kind"] != "score":
        return [lambda k, r=r: _ball_ft(r, k) for r in LEVELS[case["L"]]]
    return [lambda k, r=r: _ball_ft(r + 0.02, k) - 2.0 * _ball_ft(r, k) for r in LEVELS[case["L"]]]


def _grid(G, N):
    """P^-3 sum_m G(m) exp(2 pi i m . t / P) on t = -P/2 + P k / N (real, from the half spectrum)."""
    m = _fft_modes(N)
    sign = 1 - 2 * ((m[:, None, None] + m[None, :, None] + torch.arange(N // 2, device="cuda")) % 2)
    full = torch.zeros((N, N, N // 2 + 1), dtype=torch.complex128, device="cuda")
    full[..., : N // 2] = G * sign
    return torch.fft.irfftn(full, s=(N, N, N), norm="forward") / P ** 3


def _rotated(x, q):
    return x.double() @ _rotation(q).T


def _half_modes(N, count, canonical):
    """The lowest modes of the half space by (|m|^2, m_x, m_y, m_z): with `canonical` the half space of one mode
    per conjugate pair (0 among them), else every m != 0 with m_z >= 0."""
    top = N // 2 - 1
    c = min(top, int(math.ceil((3.0 * count / (2 * math.pi)) ** (1 / 3))) + 2)
    while True:
        r = torch.arange(-c, c + 1)
        m = torch.stack(torch.meshgrid(r, r, torch.arange(0, c + 1), indexing="ij"), dim=-1).reshape(-1, 3)
        x, y, z = m[:, 0], m[:, 1], m[:, 2]
        keep = (z > 0) | (y > 0) | ((y == 0) & (x >= 0)) if canonical else (x != 0) | (y != 0) | (z != 0)
        m = m[keep]
        q = (m ** 2).sum(1)
        if c == top or int((q <= c * c).sum()) >= count:  # no mode outside the cube is lower than these
            break
        c += 1
    b = 4 * N
    order = torch.argsort((((q * b + m[:, 0] + b // 2) * b + m[:, 1] + b // 2) * b + m[:, 2]))
    return m[order[:count]].double().cuda()


def _cone_ft(N, Nr):
    """Transform of the trimmed half-cone {|y| <= -s, -L <= s <= 0} at (|m|^2, eta): Gauss-Legendre over s."""
    t, w = np.polynomial.legendre.leggauss(160)
    s = torch.tensor(-LIFT_L * (t + 1) / 2, device="cuda")
    w = torch.tensor(w * LIFT_L / 2, device="cuda")
    k = 2 * math.pi / P * torch.arange(3 * (N // 2) ** 2 + 1, dtype=torch.float64, device="cuda").sqrt()
    ball = torch.stack([_ball_ft(-v, k) for v in s], dim=1) * w
    return ball.to(torch.complex128) @ _phases(s, _fft_modes(Nr), LIFT_PR).T


def _lift_exact(case, seed):
    N, Nr = case["N"], case["Nr"]
    m, mz, eta = _fft_modes(N), torch.arange(N // 2, dtype=torch.float64, device="cuda"), _fft_modes(Nr)
    q = (m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2).long()
    cone = _cone_ft(N, Nr)
    A, B = _lift_knots(seed, case["nA"], 4).double(), _lift_knots(seed, case["nB"], 5).double()
    xb = B[:, :3] @ _rotation(_quats(seed, 1)[0]).T
    out = [torch.zeros((N, N, N // 2), dtype=torch.complex128, device="cuda") for _ in _lift_sections(case)]

    def rho(x, r, half):
        """sum_j exp(-2 pi i (m . x_j / P + eta r_j / P_r)) for m_x in `half`, (half N, N/2 Nr)."""
        S = torch.zeros((len(half) * N, N // 2 * Nr), dtype=torch.complex128, device="cuda")
        step = max(1, (1 << 25) // max(len(half) * N, N // 2 * Nr))
        for i in range(0, x.shape[0], step):
            c, e = x[i:i + step], r[i:i + step]
            xy = (_phases(c[:, 0], half)[:, None, :] * _phases(c[:, 1], m)[None, :, :]).reshape(-1, c.shape[0])
            ze = (_phases(c[:, 2], mz)[:, None, :] * _phases(e, eta, LIFT_PR)[None, :, :]).reshape(-1, c.shape[0])
            S += xy @ ze.T
        return S.reshape(len(half), N, N // 2, Nr)
    for i in range(0, N, 32):
        G = rho(A[:, :3], A[:, 3], m[i:i + 32]) * rho(xb, -B[:, 3], m[i:i + 32]).conj() * cone[q[i:i + 32]] ** 2
        G[..., Nr // 2] = 0
        for o, r in zip(out, _lift_sections(case)):
            o[i:i + 32] = (G * _phases(torch.tensor([-r], device="cuda", dtype=torch.float64), eta, LIFT_PR)[:, 0]).sum(-1)
    for o in out:
        o[N // 2] = 0
        o[:, N // 2] = 0
    return torch.stack([_grid(o, N) / LIFT_PR for o in out])


def _mlp_exact(case, seed):
    H = case["H"]
    p, X, t = (v.double() for v in _mlp_inputs(case, seed))
    X = X[:, :132]
    sizes = [H * 132, H, H * H, H, H, 1]
    W1, b1, W2, b2, w3, b3 = torch.split(p, sizes)
    W1, W2 = W1.reshape(H, 132), W2.reshape(H, H)
    a1 = (X @ W1.T + b1).clamp_min(0)
    a2 = (a1 @ W2.T + b2).clamp_min(0)
    y = a2 @ w3 + b3
    if not case["train"]:
        return y
    d = 2 * (y - t) / len(t)
    d2 = d[:, None] * w3 * (a2 > 0)
    d1 = (d2 @ W2) * (a1 > 0)
    grads = torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ a1).reshape(-1), d2.sum(0), a2.T @ d, d.sum()[None]])
    return grads, ((y - t) ** 2).mean()[None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _mlp_exact(case, seed)
    if kind == "lifted":
        return _lift_exact(case, seed)
    N, w = case["N"], _weights(case)
    if kind == "ragged":
        shapes, peak = _ragged_shapes(case, seed), []
        for i, q in enumerate(_quats(seed, case["pairs"])):
            (xa, la), (xb, lb) = ((x.cuda(), l.cuda()) for x, l in shapes[2 * i:2 * i + 2])
            G = _spectrum(xa.double(), la, N, w) * _spectrum(_rotated(xb, q), lb, N, w).conj()
            peak.append(_grid(G, N).max())
        return torch.stack(peak), None
    if kind == "moments":
        g = _gen(seed, 2)
        x = _torus(g, case["nA"])
        lev = _levels(g, case["nA"], case["L"]).long()
        m = _half_modes(N, 64, False)
        radii = torch.tensor(LEVELS[case["L"]], dtype=torch.float64, device="cuda")
        k = 2 * math.pi / P * m.norm(dim=1)
        h = torch.stack([_ball_ft(r, k) for r in radii])  # (L, 64)
        f0 = (4 * math.pi / 3 * radii[lev] ** 3).sum()
        rows = []
        for q in _quats(seed, case["k"]):
            a = m @ (_rotated(x, q).T / P)
            a = -2 * math.pi * (a - a.round())
            v = h[lev].T
            rows.append(torch.hypot((a.cos() * v).sum(1), (a.sin() * v).sum(1)) / f0)
        return torch.stack(rows)
    (xa, la), (xb, lb) = _two_shapes(case, seed)
    FA = _spectrum(xa.double(), la, N, w)
    if kind == "query":
        G = FA * _spectrum(_rotated(xb, _quats(seed, 1)[0]), lb, N, w).conj()
        m = _half_modes(N, min(case["modes"], ((N - 1) ** 3 + 1) // 2), True)
        v = G[m[:, 0].long(), m[:, 1].long(), m[:, 2].long()] * torch.where((m == 0).all(1), 1.0, 2.0)
        t, out = _u(_gen(seed, 6), case["pts"], 3) * P - P / 2, []
        for c in t.double().split(1024):
            a = m @ c.T / P
            a = 2 * math.pi * (a - a.round())
            out.append((v.real[:, None] * a.cos() - v.imag[:, None] * a.sin()).sum(0) / P ** 3)
        return torch.cat(out)
    grids = []
    for q in _pair_quats(case, seed):
        G = FA * _spectrum(_rotated(xb, q), lb, N, w).conj()
        grids.append(_grid(-G if kind == "score" else G, N))
        if kind == "sweep":
            grids[-1] = grids[-1].max()
    return (torch.stack(grids), None) if kind == "sweep" else torch.stack(grids)
