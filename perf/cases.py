"""The work that a user of this library has it do, as cases of one measurement.

A case is one pass through the public Python entry points: a whole solve of a
cube (plain MUFFIN, or ADA-PT with its two chain groups), the single
operators, what happens before a first iteration, or a small served stream.
Inputs are drawn on the GPU from a seed with the recipe of ``synth`` (point
sources and blobs with power-law spectra, a uv coverage per band, 20 dB SNR).
``exact`` restates the iteration in 64 bits with plain torch.

``kind`` is one of
  solve      ``Plan.solve`` from X0 = 0 on a plan that the user keeps
  tune       ``Plan.sure_tune`` (ADA-PT, six chains) from X0 = 0
  operators  the four operators on one cube (gradient with a dirty cube)
  setup      new PSFs, noise estimate, weights and objective of a cube
  serve      requests of uneven shapes through ``Server``
"""
import math

import numpy as np
import torch

import paper_1905_08468_gb300 as muffin


def _case(name, kind, n, bands, iters=0, **more):
    c = {"name": name, "kind": kind, "n": n, "bands": bands, "iters": iters, "batch": 1,
         "wavelets": 8, "levels": 3, "dictionary": "daubechies", "precision": "tf32"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest documented workload: a quick look at one field, bound
        # by launches and latency
        _case("plain-64x8", "solve", 64, 8, 200),
        # the ordinary cube of the paper's size class per node
        _case("plain-256x32", "solve", 256, 32, 100),
        # many channels, all duals resident: the large single cube at half its side
        _case("plain-1024x256", "solve", 1024, 256, 15),
        # an odd channel count (flagged channels dropped), fewer bases, four levels
        _case("ragged-256x37", "solve", 256, 37, 50, wavelets=5, levels=4),
        # the caller asks for the spectral step in FP32
        _case("fp32-512x128", "solve", 512, 128, 20, precision="fp32"),
        # a pool of small cubes advanced by the same launches
        _case("batch-8x128x16", "solve", 128, 16, 50, batch=8),
        # weight tuning on the ordinary cube (the convergence study's shape)
        _case("tune-256x32", "tune", 256, 32, 50, window=10),
        # weight tuning on the large benchmark cube
        _case("tune-1024x64", "tune", 1024, 64, 20, window=10),
        # weight tuning with the starlet in place of the wavelet union
        _case("starlet-tune-512x32", "tune", 512, 32, 20, window=10, dictionary="iuwt"),
        # the operators alone, as a caller's own iteration or check uses them
        _case("operators-512x48", "operators", 512, 48),
        # what comes before the first iteration on a new pointing
        _case("setup-512x64", "setup", 512, 64),
        # uneven requests arriving together at a server
        _case("serve-mix", "serve", 256, 32, 60, requests=6),
    ]


# work of a pass in voxels x iterations x chains, above which draws are not made
_MOST = 1024 * 1024 * 64 * 6 * 20


def draw(rng):
    while True:
        kind = rng.choice(["solve", "solve", "solve", "tune", "tune", "operators", "setup", "serve"])
        n = 1 << rng.randint(4, 10)
        bands = int(round(math.exp(rng.uniform(math.log(2), math.log(256)))))
        c = _case("", kind, n, bands, int(round(math.exp(rng.uniform(math.log(8), math.log(150))))))
        del c["name"]
        if kind in ("solve", "tune"):
            c["dictionary"] = rng.choice(["daubechies", "daubechies", "daubechies", "iuwt"])
            c["levels"] = rng.randint(1, 4)
            c["wavelets"] = rng.choice([1, 2, 4, 6, 8, 8, 8])
            c["precision"] = rng.choice(["tf32", "tf32", "fp32"])
        if kind == "solve":
            c["batch"] = rng.choice([1, 1, 2, 3, 8])
        if c["precision"] == "fp32" or rng.random() < 0.5:
            c["bands"] = 1 << max(1, int(round(math.log2(bands))))
        if kind == "tune":
            c["window"] = rng.choice([5, 7, 10])
        if kind == "serve":
            c["requests"] = rng.randint(2, 8)
            c["n"], c["bands"], c["iters"] = 256, 32, rng.randint(20, 100)
        voxels = c["n"] ** 2 * c["bands"] * c["batch"]
        if voxels > 1024 * 1024 * 64:
            continue
        if 2 * voxels * max(10, c["iters"]) * (6 if kind == "tune" else 1) <= _MOST:
            return c


# ---------------------------------------------------------------- inputs
def _cube(n, bands, seed):
    """psf, dirty, delta [L][n][n] float32 on the GPU and the noise variances."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def rand(*s):
        return torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)

    nu = 1 + torch.arange(bands, device="cuda", dtype=torch.float64) / max(1, bands - 1)
    amp = torch.exp(rand(n, n) * math.log(10) - math.log(10)) * (rand(n, n) < 200 / 256 ** 2)
    slope = 2 * rand(n, n) - 1
    blobs = max(1, round(20 * n * n / 65536))
    centre, width, tilt = n * rand(2, blobs), 2 + 3 * rand(blobs), 2 * rand(blobs) - 1
    d = (torch.arange(n, device="cuda", dtype=torch.float64) - centre[..., None]).abs()
    g = torch.exp(-0.5 * (torch.minimum(d, n - d) / width[:, None]) ** 2)
    uv = 0.15 * torch.randn(2, max(100, round(20000 * n * n / 65536)), generator=gen, device="cuda",
                            dtype=torch.float64)
    psf = torch.empty(bands, n, n, device="cuda")
    dirty = torch.empty_like(psf)
    var = np.empty(bands)
    for k in range(bands):
        f = float(nu[k])
        sky = amp * f ** slope + (g[0] * (0.3 * f ** tilt)[:, None]).T @ g[1]
        q = uv * f
        q = torch.round(q[:, (q.abs() < 0.5).all(0)] * n).long()
        at = torch.cat([(q[0] % n) * n + q[1] % n, (-q[0] % n) * n + (-q[1]) % n])
        p = torch.fft.ifft2(torch.bincount(at, minlength=n * n).double().view(n, n)).real
        psf[k] = p / p[0, 0]
        hx = torch.fft.irfft2(torch.fft.rfft2(psf[k].double()) * torch.fft.rfft2(sky), s=(n, n))
        var[k] = float((hx * hx).mean()) / 100
        dirty[k] = hx + math.sqrt(var[k]) * torch.randn(n, n, generator=gen, device="cuda",
                                                        dtype=torch.float64)
    delta = torch.randn(bands, n, n, generator=gen, device="cuda")
    return psf, dirty, delta, var


def _theta(case, seed):
    """(mu, gamma) in the range around the convergence study's optimum."""
    r = np.random.default_rng(seed)
    return tuple(float(v) for v in np.exp(r.uniform(math.log(5e-3), math.log(2e-2), 2)))


def _requests(case, seed):
    """Shapes of a served mix: sides and bands of the served stream."""
    r = np.random.default_rng(7 * case["requests"] + case["iters"])
    return [(int(n), int(b)) for n, b in zip(r.choice([128, 256], case["requests"]),
                                             r.choice([16, 32, 64], case["requests"]))]


def _tuning(case, var):
    vox = case["n"] ** 2 * case["bands"]
    return dict(window=case["window"], eta=(0.2 / vox, 2.0 / vox),
                eps=0.1 * math.sqrt(float(np.mean(var))))


def prepare(case, seed):
    n, bands, batch = case["n"], case["bands"], case["batch"]
    s = {"case": case, "theta": _theta(case, seed)}
    if case["kind"] == "serve":
        s["server"] = muffin.Server()
        s["jobs"] = []
        for i, (m, b) in enumerate(_requests(case, seed)):
            psf, dirty, _, _ = _cube(m, b, 1000 * seed + i)
            s["jobs"].append((psf.cpu().numpy(), dirty.cpu().numpy(), np.empty((b, m, m), np.float32)))
        return s
    cubes = [_cube(n, bands, 1000 * seed + i) for i in range(batch)]
    s["psf"], s["dirty"], s["delta"] = (torch.cat([c[i] for c in cubes]) for i in range(3))
    s["var"] = np.concatenate([c[3] for c in cubes])
    s["plan"] = muffin.Plan(n, bands, s["psf"], n_wavelets=case["wavelets"], levels=case["levels"],
                            dictionary=case["dictionary"], precision=case["precision"], batch=batch,
                            sure=case["kind"] == "tune")
    if case["kind"] == "operators":
        s["u"] = torch.randn(bands, 8, n, n, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    case, (mu, gamma) = state["case"], state["theta"]
    kind = case["kind"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(p, d, mu, gamma, case["iters"]) for p, d, _ in state["jobs"]]
        left = dict(enumerate(tickets))
        while left:
            server.step()
            for i, t in list(left.items()):
                if server.poll(t, state["jobs"][i][2]):
                    del left[i]
        return [out for _, _, out in state["jobs"]]
    plan, dirty = state["plan"], state["dirty"]
    x = torch.zeros_like(dirty)
    if kind == "solve":
        info = plan.solve(dirty, x, case["iters"], mu, gamma)
        return {"x": x, "tau": info.tau}
    if kind == "tune":
        theta, trace, _ = plan.sure_tune(dirty, state["delta"], state["var"], x, (mu, gamma),
                                         case["iters"], **_tuning(case, state["var"]))
        return {"x": x, "theta": list(theta)}
    if kind == "operators":
        u, v = torch.empty_like(state["u"]), torch.empty_like(dirty)
        out = {"u": u, "v": v, "g": torch.empty_like(dirty), "x": x, "t": torch.empty_like(dirty)}
        plan.op_gradient(state["delta"], out["g"], dirty)
        plan.op_analysis(dirty, u)
        plan.op_synthesis(state["u"], x)
        plan.op_dct(dirty, v)
        plan.op_dct(v, out["t"], inverse=True)
        return out
    plan.load_psf(state["psf"])
    alpha, beta = plan.weights_from_x0(dirty, 1e-2, 1e-2)
    return {"lipschitz": plan.lipschitz, "alpha": alpha, "beta": beta,
            "noise": plan.noise_mad(dirty), "objective": plan.objective(dirty, dirty.abs(), mu, gamma)}


# ---------------------------------------------------------------- what a pass needs
def _planes(case):
    return case["levels"] + 1 if case["dictionary"] == "iuwt" else case["wavelets"]


def _flops(n, bands, planes, levels, dictionary):
    """Of one iteration of one chain, a voxel: filters both ways, FFTs, DCT pair."""
    if dictionary == "iuwt":
        w = 2 * 20 * levels
    else:
        w = 2 * 8 * sum(range(1, planes + 1)) * sum(0.25 ** j for j in range(levels))
    return w + 10 * math.log2(n) + 5 * math.log2(max(2, bands)) + 12


def work(case):
    n, bands = case["n"], case["bands"]
    vox = n * n * bands * case["batch"]
    k, kind = _planes(case), case["kind"]
    if kind == "serve":
        parts = [work(_case("", "solve", m, b, case["iters"])) for m, b in _requests(case, 0)]
        return {q: sum(p[q] for p in parts) for q in ("bytes", "flops")}
    f = _flops(n, bands, k, case["levels"], case["dictionary"])
    if kind == "solve":     # x, v and the planes of u, read and written; b and |h|^2 read
        return {"bytes": vox * (8 + case["iters"] * (16 + 8 * k + 6)), "flops": vox * case["iters"] * f}
    if kind == "tune":
        return {"bytes": vox * (12 + case["iters"] * (6 * (16 + 8 * k) + 10)),
                "flops": vox * case["iters"] * 6 * f}
    if kind == "operators":  # gradient 14, analysis and synthesis 4 + 4k, two DCTs 8
        return {"bytes": vox * (14 + 2 * (4 + 4 * k) + 16), "flops": vox * 2 * f}
    return {"bytes": vox * 4 * 4, "flops": vox * 2 * f}   # psf and the cubes read


# ---------------------------------------------------------------- 64 bits
def _lowpass(p):
    """Minimum-phase Daubechies filter of p vanishing moments."""
    roots = []
    poly = [math.comb(p - 1 + j, j) for j in range(p)][::-1]
    for y in np.roots(poly):
        r = np.sqrt(y * y - y + 0j)
        z = 1 - 2 * y + 2 * r
        roots.append(z if abs(z) < 1 else 1 - 2 * y - 2 * r)
    h = np.real(np.poly([-1.0] * p + roots))
    return h * (math.sqrt(2) / h.sum())


def _down(x, h, dim):
    """a[k] = sum_i h[i] x[(2k + i) mod M] along dim."""
    m = x.shape[dim]
    at = torch.arange(0, m, 2, device=x.device)
    out = x.index_select(dim, at) * float(h[0])
    for i, c in enumerate(h[1:], 1):
        out.add_(x.index_select(dim, (at + i) % m), alpha=float(c))
    return out


def _up(a, h, dim):
    """The transpose of _down: x[2k + e] = sum_s h[2s + e] a[k - s]."""
    half = [a * float(h[e]) for e in (0, 1)]
    for s in range(1, len(h) // 2):
        r = a.roll(s, dim)
        for e in (0, 1):
            half[e].add_(r, alpha=float(h[2 * s + e]))
    shape = list(a.shape)
    shape[dim] *= 2
    return torch.stack(half, -1 if dim == -1 else -2).reshape(shape)


def _smooth(x, j):
    for dim in (-1, -2):
        x = sum(w / 16 * x.roll(s << j, dim) for w, s in ((1, -2), (4, -1), (6, 0), (4, 1), (1, 2)))
    return x


class _Exact:
    """W, W^T, C and H^T H of a plan in 64 bits, on one band axis."""

    def __init__(self, case):
        self.c, self.k = case, _planes(case)
        lo = [_lowpass(p) for p in range(1, case["wavelets"] + 1)]
        self.taps = [(h, [(-1) ** i * h[-1 - i] for i in range(len(h))]) for h in lo]
        self.norm2 = 1.0 if case["dictionary"] == "iuwt" else float(case["wavelets"])
        b = case["bands"]
        i = torch.arange(b, device="cuda", dtype=torch.float64)
        self.C = torch.cos(math.pi * (i[None] + 0.5) * i[:, None] / b) * math.sqrt(2 / b)
        self.C[0] /= math.sqrt(2)

    def analysis(self, x, k):
        """Plane k of W x."""
        if self.c["dictionary"] == "iuwt":
            for j in range(k):
                x = _smooth(x, j)
            return x - _smooth(x, k) if k < self.k - 1 else x
        h, g = self.taps[k]
        out, ll = torch.empty_like(x), x
        for _ in range(self.c["levels"]):
            m = ll.shape[-1] // 2
            lo, hi = _down(ll, h, -1), _down(ll, g, -1)
            out[:, :m, m:2 * m], out[:, m:2 * m, m:2 * m] = _down(hi, h, -2), _down(hi, g, -2)
            out[:, m:2 * m, :m] = _down(lo, g, -2)
            ll = _down(lo, h, -2)
        out[:, :ll.shape[-2], :ll.shape[-1]] = ll
        return out

    def synthesis(self, u, k):
        """W_k^T u of plane k."""
        if self.c["dictionary"] == "iuwt":
            u = u - _smooth(u, k) if k < self.k - 1 else u
            for j in range(k):
                u = _smooth(u, j)
            return u
        h, g = self.taps[k]
        m = u.shape[-1] >> self.c["levels"]
        ll = u[:, :m, :m]
        for _ in range(self.c["levels"]):
            lo = _up(ll, h, -2) + _up(u[:, m:2 * m, :m], g, -2)
            hi = _up(u[:, :m, m:2 * m], h, -2) + _up(u[:, m:2 * m, m:2 * m], g, -2)
            ll = _up(lo, h, -1) + _up(hi, g, -1)
            m *= 2
        return ll

    def dct(self, z, inverse=False):
        m = self.C.T if inverse else self.C
        return (m @ z.reshape(z.shape[0], -1)).view_as(z)


def _hth(power, x):
    return torch.fft.irfft2(power * torch.fft.rfft2(x), s=x.shape[-2:])


def _iterate(E, power, b, tau, mu, gamma, s, sigma=10.0):
    """One iteration of a chain group: primal, and with ADA-PT d/dmu, d/dgamma.
    s: x [C], u [C][K], v [C], t [C]."""
    C = len(s["x"])
    old = s["x"]
    syn = [sum(E.synthesis(s["u"][c][k], k) for k in range(E.k)) for c in range(C)]
    dual = [mu * syn[0]] + ([syn[0] + mu * syn[1], mu * syn[2]] if C == 3 else [])
    m = [old[c] - tau * (_hth(power, old[c]) - (b if c == 0 else 0) + dual[c] + s["t"][c]) for c in range(C)]
    del syn, dual
    keep = m[0] > 0
    new = [torch.where(keep, q, 0.0) for q in m]
    z = [2 * p - q for p, q in zip(new, old)]
    w, q = z[:], [sigma * mu, sigma, sigma * mu]
    if C == 3:
        w[1] = z[0] + mu * z[1]
    for k in range(E.k):
        p = [s["u"][c][k] + q[c] * E.analysis(w[c], k) for c in range(C)]
        keep = p[0].abs() <= 1
        s["u"][0][k] = p[0].clamp(-1, 1)
        for c in range(1, C):
            s["u"][c][k] = torch.where(keep, p[c], 0.0)
    p = [s["v"][c] + sigma * (gamma if c < 2 else 1.0) * E.dct(z[c] if c < 2 else z[0] + gamma * z[2])
         for c in range(C)]
    keep = p[0].abs() <= 1
    s["v"] = [p[0].clamp(-1, 1)] + [torch.where(keep, r, 0.0) for r in p[1:]]
    s["t"] = [gamma * E.dct(r, True) for r in s["v"][:2]]
    if C == 3:
        s["t"].append(E.dct(gamma * s["v"][2] + s["v"][0], True))
    s["x"] = new


def _start(E, like, C):
    zero = lambda: torch.zeros_like(like)  # noqa: E731
    return {"x": [zero() for _ in range(C)], "v": [zero() for _ in range(C)], "t": [zero() for _ in range(C)],
            "u": [[zero() for _ in range(E.k)] for _ in range(C)]}


def _exact_solve(case, cube, theta):
    psf, dirty, delta, var = cube
    E = _Exact(case)
    n, bands, sigma = case["n"], case["bands"], 10.0
    H = torch.fft.rfft2(psf.double())
    power = H.abs() ** 2
    mu, gamma = theta
    adj = lambda y: torch.fft.irfft2(H.conj() * torch.fft.rfft2(y.double()), s=(n, n))  # noqa: E731
    tau_of = lambda m, g: 0.99 / (0.5 * float(power.max())  # noqa: E731
                                  + sigma * (E.norm2 * bands * m * m + n * n * g * g))
    b = adj(dirty)
    tune = case["kind"] == "tune"
    groups = [_start(E, b, 3 if tune else 1) for _ in range(2 if tune else 1)]
    data = [b]
    if tune:
        opt = _tuning(case, var)
        probe = adj(delta)
        data.append(b + opt["eps"] * probe)
        weight = torch.from_numpy(2 * var / opt["eps"]).cuda()
    tau = tau_of(mu, gamma)
    for it in range(1, case["iters"] + 1):
        for s, d in zip(groups, data):
            _iterate(E, power, d, tau, mu, gamma, s)
        if tune and it % opt["window"] == 0:
            x, y = groups[0]["x"], groups[1]["x"]
            grad = _hth(power, x[0]) - b
            sugar = [float(2 * (grad * x[c]).sum() + (weight * ((y[c] - x[c]) * probe).sum((1, 2))).sum())
                     for c in (1, 2)]
            mu = max(mu - opt["eta"][0] * sugar[0], 1e-8)
            gamma = max(gamma - opt["eta"][1] * sugar[1], 1e-8)
            tau = tau_of(mu, gamma)
            for s in groups:
                s["x"][1:], s["v"][1:], s["t"][1:] = ([torch.zeros_like(b) for _ in range(2)] for _ in range(3))
                s["u"][1:] = [[torch.zeros_like(b) for _ in range(E.k)] for _ in range(2)]
    return groups[0]["x"][0], (mu, gamma), tau


def exact(case, seed):
    n, bands, kind = case["n"], case["bands"], case["kind"]
    mu, gamma = theta = _theta(case, seed)
    if kind == "serve":
        return [_exact_solve(_case("", "solve", m, b, case["iters"]), _cube(m, b, 1000 * seed + i), theta)[0]
                for i, (m, b) in enumerate(_requests(case, seed))]
    cost = n * n * bands * case["batch"] * max(1, case["iters"]) * (6 if kind == "tune" else 1) * _planes(case)
    small = 0.002 * case["iters"] * case["batch"] * _planes(case) * case["levels"] * (6 if kind == "tune" else 1)
    if cost > 7e10 or small > 30:
        return None       # many minutes in 64 bits
    if kind in ("solve", "tune"):
        got = [_exact_solve(case, _cube(n, bands, 1000 * seed + i), theta) for i in range(case["batch"])]
        x = torch.cat([g[0] for g in got])
        return {"x": x, "theta": list(got[0][1])} if kind == "tune" else {"x": x, "tau": got[0][2]}
    E = _Exact(case)
    psf, dirty, delta, _ = _cube(n, bands, 1000 * seed)
    H, y = torch.fft.rfft2(psf.double()), dirty.double()
    if kind == "operators":
        u = torch.randn(bands, 8, n, n, device="cuda", generator=torch.Generator("cuda").manual_seed(seed)).double()
        v = E.dct(y)
        res = H * torch.fft.rfft2(delta.double()) - torch.fft.rfft2(y)
        return {"u": torch.stack([E.analysis(y, k) for k in range(E.k)], 1), "v": v,
                "g": torch.fft.irfft2(H.conj() * res, s=(n, n)),
                "x": sum(E.synthesis(u[:, k], k) for k in range(E.k)), "t": E.dct(v, True)}
    alpha = 1 / (y.square().sum(0).sqrt() + 1e-2)
    beta = 1 / (math.sqrt(E.norm2) * y.square().sum((1, 2)).sqrt() + 1e-2)
    a = y.abs()
    spatial = sum(E.analysis(a, k).abs().sum((1, 2)) for k in range(E.k))
    fit = (torch.fft.irfft2(H * torch.fft.rfft2(a), s=(n, n)) - y).square().sum()
    cost = 0.5 * fit + mu * (beta * spatial).sum() + gamma * (alpha * E.dct(a).abs()).sum()
    d = (y[:, ::2, ::2] - y[:, ::2, 1::2] - y[:, 1::2, ::2] + y[:, 1::2, 1::2]) / 2


    def middle(v):
        v = v.flatten(1).sort(1).values
        m = v.shape[1]
        return (v[:, (m - 1) // 2] + v[:, m // 2]) / 2
    noise = (middle((d - middle(d)[:, None, None]).abs()) / 0.6744897501960817) ** 2
    return {"lipschitz": float(H.abs().max() ** 2), "alpha": alpha, "beta": beta, "noise": noise,
            "objective": float(cost)}
