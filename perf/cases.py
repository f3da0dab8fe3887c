"""The work that programs have this library do, as cases that can be timed and compared.

A case is one call of the public binding (``paper_1412_8398_gb300.fftls`` / ``warmstart``) on inputs that
``prepare`` makes from a seed: periodised Boolean images of spheres (discs in 2D), the microstructures of the
repository's configurations, tests and benchmark.  The solver cases keep one handle for all their calls, as a
parametric study does: every call has a new image, so nothing but workspaces and tile schedules carries over.

What the solver computes in single precision (``fp32``, and the fields of the ``fp32_refine64`` ladder, whose
iterates are single-precision corrections stopped at the tolerance) the program keeps in single precision; the
results of ``fp64`` solves stay as they are.

``exact`` restates eq. (ds) / (as) of the paper in plain torch in 64 bits (and the warm start's network as sums of
shifted matrix products), without this repository's code.
"""
import math

import numpy as np
import torch

from paper_1412_8398_gb300 import fftls, warmstart

_SOLVER = None


def _solver():
    global _SOLVER
    if _SOLVER is None:
        _SOLVER = fftls.Solver(0)
    return _SOLVER


def listed():
    return [
        # The smallest call: a 24^3 double-precision solve from host arrays into host arrays (the library's defaults).
        dict(name="cube_24_fp64_host", kind="solve", n1=24, n2=24, n3=24, radius=3.0, fraction=0.3, contrast=10.0,
             green="R", scheme="AS", precision="fp64", stop="eta", tol=1e-8, max_iter=1000, about=45, host=True),
        # 2D: discs of 100 times the matrix's stiffness under shear, the direct scheme to its default tolerance.
        dict(name="disc2d_128_ds_fp64", kind="solve", n1=128, n2=128, n3=0, radius=12.0, fraction=0.25,
             contrast=100.0, green="R", scheme="DS", precision="fp64", stop="eta", tol=1e-8, max_iter=5000, about=900,
             host=False),
        # The smallest grid of the batched study, alone: a ladder solve where latency and launches count.
        dict(name="cube_32_ladder", kind="solve", n1=32, n2=32, n3=32, radius=4.0, fraction=0.3, contrast=100.0,
             green="R", scheme="AS", precision="fp32_refine64", stop="eta", tol=1e-6, max_iter=3000, about=100,
             host=False),
        # The field-accuracy studies in 2D: 512^2, contrast 1000, accelerated, stopped on the largest field change.
        dict(name="cell2d_512_maxdelta", kind="solve", n1=512, n2=512, n3=0, radius=40.0, fraction=0.25,
             contrast=1000.0, green="R", scheme="AS", precision="fp64", stop="maxdelta", tol=1e-9, max_iter=5000,
             about=600, host=False),
        # The paper's 64^3 Boolean model (spheres of diameter 5, 17 %) in double precision.
        dict(name="cube_64_fp64", kind="solve", n1=64, n2=64, n3=64, radius=2.5, fraction=0.17, contrast=10.0,
             green="R", scheme="AS", precision="fp64", stop="eta", tol=1e-8, max_iter=1000, about=45, host=False),
        # A tomography cut: no two sides alike, none a power of two, centred differences.
        dict(name="ragged_100x90x75_c_ladder", kind="solve", n1=100, n2=90, n3=75, radius=6.0, fraction=0.3,
             contrast=30.0, green="C", scheme="AS", precision="fp32_refine64", stop="eta", tol=1e-6, max_iter=3000,
             about=60, host=False),
        # A statistical study: independent samples of uneven sizes (32^3 to 128^3) solved together by the ladder.
        dict(name="batched_24_ladder", kind="batched", count=24, tol=1e-6, precision="fp32_refine64", max_iter=3000,
             about=100),
        # The reference operator G of Moulinec and Suquet on the 128^3 configuration, with the stress field.
        dict(name="cube_128_ms_ladder", kind="solve", n1=128, n2=128, n3=128, radius=6.0, fraction=0.3, contrast=10.0,
             green="MS", scheme="AS", precision="fp32_refine64", stop="eta", tol=1e-6, max_iter=3000, about=40,
             host=False),
        # Forward / backward differences under the direct scheme on the same configuration.
        dict(name="cube_128_w_ds_ladder", kind="solve", n1=128, n2=128, n3=128, radius=6.0, fraction=0.3,
             contrast=10.0, green="W", scheme="DS", precision="fp32_refine64", stop="eta", tol=1e-6, max_iter=3000,
             about=70, host=False),
        # A whole ladder solve to tolerance at the size of the warm-start study.
        dict(name="cube_256_r_ladder", kind="solve", n1=256, n2=256, n3=256, radius=6.0, fraction=0.25, contrast=100.0,
             green="R", scheme="AS", precision="fp32_refine64", stop="eta", tol=1e-6, max_iter=3000, about=110,
             host=False),
        # The benchmark's grid: the modulus history over the first iterations at contrast 1000 (FP32).
        dict(name="cube_512_r_fp32", kind="solve", n1=512, n2=512, n3=512, radius=8.0, fraction=0.25, contrast=1000.0,
             green="R", scheme="AS", precision="fp32", stop="eta", tol=0.0, max_iter=20, about=20, host=False),
        # The warm start's network (tensor-core path) on a 256^3 image, before a warm-started solve.
        dict(name="warm_256_forward", kind="warm", n1=256, n2=256, n3=256, radius=6.0, fraction=0.25, contrast=100.0),
    ]


def _smooth(lo, hi):
    """Supported grid lengths (prime factors 2, 3, 5) in lo .. hi."""
    def ok(v):
        for p in (2, 3, 5):
            while v % p == 0:
                v //= p
        return v == 1
    return [v for v in range(lo, hi + 1) if ok(v)]


def _near(rng, lo, hi):
    """A supported length, uniform in the logarithm over lo .. hi."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_smooth(lo, hi), key=lambda v: abs(math.log(v / x)))


def draw(rng):
    u = rng.random()
    if u < 0.1:
        return dict(kind="batched", count=rng.randint(6, 24), tol=1e-6, precision="fp32_refine64", max_iter=1000,
                    about=100)
    if u < 0.2:
        n = [8 * rng.randint(4, 28) for _ in range(3)]
        return dict(kind="warm", n1=n[0], n2=n[1], n3=n[2], radius=round(rng.uniform(3, 8), 2),
                    fraction=round(rng.uniform(0.1, 0.4), 3), contrast=round(10 ** rng.uniform(1, 3), 1))
    two = u < 0.35
    precision = "fp64" if two else rng.choice(["fp64", "fp32", "fp32_refine64", "fp32_refine64"])
    scheme = rng.choice(["AS", "AS", "DS"])
    green = rng.choice(["R", "R", "C", "W", "MS"])
    if two:
        n = [_near(rng, 48, 640) for _ in range(2)] + [0]
    else:
        top = {"fp64": 128, "fp32": 400, "fp32_refine64": 200}[precision]
        n1 = _near(rng, 20, top)
        n = [n1, n1, n1] if rng.random() < 0.4 else [_near(rng, max(16, n1 // 2), min(top, 2 * n1)) for _ in range(3)]
    vox = n[0] * n[1] * max(1, n[2])
    fixed = precision == "fp32"
    cap = int(min(24 if fixed else 600, max(6, 0.2 / (vox * (0.7e-9 if precision == "fp64" else 0.09e-9)))))
    return dict(kind="solve", n1=n[0], n2=n[1], n3=n[2], radius=round(rng.uniform(2.5, 8), 2),
                fraction=round(rng.uniform(0.1, 0.4), 3),
                contrast=round(10 ** rng.uniform(0.5, 1.3 if scheme == "DS" else 3), 2), green=green, scheme=scheme,
                precision=precision, stop="eta", tol=0.0 if fixed else 1e-8 if precision == "fp64" else 1e-6,
                max_iter=cap, about=min(cap, 100), host=not fixed and vox < 40000 and rng.random() < 0.5)


def _boolean(shape, radius, fraction, seed):
    """Periodised Boolean model on the GPU: balls of one radius at seeded lattice points, uint8 image (.., n2, n1)."""
    d = len(shape)
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = int(math.floor(radius))
    ax = torch.arange(-r, r + 1, device="cuda")
    off = torch.stack(torch.meshgrid(*[ax] * d, indexing="ij"), -1).reshape(-1, d)
    off = off[(off * off).sum(1) <= radius * radius]
    count = max(1, round(-math.log(1.0 - fraction) / off.shape[0] * math.prod(shape)))
    img = torch.zeros(math.prod(shape), dtype=torch.uint8, device="cuda")
    size = torch.tensor(shape, device="cuda")
    stride = torch.tensor([math.prod(shape[i + 1:]) for i in range(d)], device="cuda")
    at = (torch.rand((count, d), generator=g, device="cuda", dtype=torch.float64) * size).long()
    for c in at.split(4096):
        img[(torch.remainder(c[:, None, :] + off, size) * stride).sum(-1).reshape(-1)] = 1
    return img.reshape(shape)


def _shape(case):
    return ((case["n3"],) if case["n3"] else ()) + (case["n2"], case["n1"])


def _phases(contrast):
    """(lambda, mu) of the matrix (E = 1, nu = 0.3) and the inclusions (E = contrast, nu = 0.2)."""
    lame = [(E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))) for E, nu in ((1.0, 0.3), (contrast, 0.2))]
    return np.array([a for a, _ in lame]), np.array([b for _, b in lame])


def _load(d, seed):
    """A macroscopic strain tensor: tension along x1 and a seeded shear."""
    e = np.zeros((d, d))
    e[0, 0] = 1.0
    e[0, 1] = e[1, 0] = 0.1 * (1 + seed % 5)
    return e


_BATCH_LENGTHS = (32, 48, 64, 96, 128)


def _batch_specs(case, seed):
    """Samples of the statistical study: every length in turn, radius 3-8, fraction 0.1-0.4, contrast 10-1000."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["count"]):
        L = _BATCH_LENGTHS[i % len(_BATCH_LENGTHS)]
        out.append((L, rng.uniform(3, 8), rng.uniform(0.1, 0.4), 10 ** rng.uniform(1, 3), int(rng.integers(1 << 30))))
    return out


# The network: (name, input channels, output channels, kernel size), as the warm start declares it.
_NET = [("enc0", 2, 8, 3), ("enc1a", 8, 16, 3), ("enc1b", 16, 16, 3), ("enc2a", 16, 32, 3), ("enc2b", 32, 32, 3),
        ("enc3a", 32, 64, 3), ("enc3b", 64, 64, 3), ("dec2", 64, 32, 3), ("dec1", 32, 16, 3), ("dec0", 16, 8, 1),
        ("out", 8, 6, 3)]


def _weights(seed):
    rng = np.random.default_rng(seed)
    return {name: ((rng.standard_normal((co, ci, k, k, k)) * math.sqrt(2.0 / (ci * k ** 3))).astype(np.float32),
                   (0.1 * rng.standard_normal(co)).astype(np.float32)) for name, ci, co, k in _NET}


def prepare(case, seed):
    if case["kind"] == "batched":
        samples = []
        for L, radius, fraction, contrast, s in _batch_specs(case, seed):
            lam, mu = _phases(contrast)
            samples.append(dict(phase=_boolean((L, L, L), radius, fraction, s), lam=lam, mu=mu, eps_bar=_load(3, s)))
        return dict(case=case, solver=_solver(), samples=samples)
    phase = _boolean(_shape(case), case["radius"], case["fraction"], seed)
    if case["kind"] == "warm":
        net = warmstart.WarmNet(0)
        net.load_arrays(_weights(seed))
        return dict(case=case, net=net, phase=phase)
    lam, mu = _phases(case["contrast"])
    return dict(case=case, solver=_solver(), phase=phase.cpu().numpy() if case["host"] else phase, lam=lam, mu=mu,
                eps_bar=_load(phase.ndim, seed))


def run(state):
    case = state["case"]
    if case["kind"] == "warm":
        return state["net"].forward_tc(state["phase"], case["contrast"])
    if case["kind"] == "batched":
        res, _ = state["solver"].solve_batched(state["samples"], tol=case["tol"], max_iter=case["max_iter"],
                                               precision=case["precision"], want_strain=True, device_outputs=True)
        return dict(strain=[r.strain.float() for r in res],
                    mean_stress=np.stack([r.mean_stress for r in res]).astype(np.float32))
    r = state["solver"].solve(state["phase"], state["lam"], state["mu"], state["eps_bar"], green=case["green"],
                              scheme=case["scheme"], precision=case["precision"], stop=case["stop"], tol=case["tol"],
                              max_iter=case["max_iter"], want_stress=case["precision"] == "fp64")
    if case["precision"] == "fp64":
        return dict(strain=r.strain, stress=r.stress, mean_stress=r.mean_stress, mean_strain=r.mean_strain)
    out = dict(strain=r.strain.astype(np.float32) if case["host"] else r.strain.float(),
               mean_stress=r.mean_stress.astype(np.float32), mean_strain=r.mean_strain.astype(np.float32))
    if case["tol"] == 0.0:  # a fixed number of iterations: the histories are what is asked for
        out["eta"] = r.eta_history.astype(np.float32)
        out["modulus"] = r.mean_stress_history.astype(np.float32)
    return out


def work(case):
    """Bytes: the image and the result once, and the strain iterate read and written once an iteration (`about`
    iterations).  Flops: the forward and inverse real transforms of every strain component (2.5 N log2 N each) and
    about 30 an iteration per voxel and component for the phases' law, the Green operator, the norm and the update."""
    if case["kind"] == "warm":
        n = case["n1"] * case["n2"] * case["n3"]
        level = dict(enc1a=1, enc1b=1, enc2a=2, enc2b=2, enc3a=3, enc3b=3, dec2=2, dec1=1)
        return {"bytes": n * (1 + 24), "flops": sum(2 * ci * co * k ** 3 * (n >> (3 * level.get(name, 0)))
                                                    for name, ci, co, k in _NET)}
    if case["kind"] == "batched":
        one = [work(dict(kind="solve", n1=L, n2=L, n3=L, precision=case["precision"], about=case["about"]))
               for L in (_BATCH_LENGTHS[i % len(_BATCH_LENGTHS)] for i in range(case["count"]))]
        return {"bytes": sum(w["bytes"] for w in one), "flops": sum(w["flops"] for w in one)}
    n, nc = case["n1"] * case["n2"] * max(1, case["n3"]), 6 if case["n3"] else 3
    size, fields = (8, 2) if case["precision"] == "fp64" else (4, 1)
    return {"bytes": n * (1 + fields * nc * size + case["about"] * 2 * nc * size),
            "flops": case["about"] * n * nc * (5 * math.log2(n) + 30)}


# ---------------------------------------------------------------------------
# 64-bit restatement
# ---------------------------------------------------------------------------
def _exact_solve(phase, lam, mu, eps_bar, green, scheme, tol, max_iter, stop):
    """eq. (ds) / (as) in 64 bits with torch's FFTs; (strain, stress, mean stress, mean strain, histories)."""
    d = phase.ndim
    shape = tuple(phase.shape)
    N = phase.numel()
    IJ = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)] if d == 3 else [(0, 0), (1, 1), (0, 1)]
    full = green == "MS"  # operator G treats both sides of the spectrum alike only on the full one
    axes = tuple(range(1, d + 1))
    ids = phase.long()
    lf, mf = torch.tensor(lam, device="cuda")[ids], torch.tensor(mu, device="cuda")[ids]
    kap = lam + 2.0 / d * mu
    k0, m0 = ((math.sqrt(kap.min() * kap.max()), math.sqrt(mu.min() * mu.max())) if scheme == "AS" else
              (0.5 * (kap.min() + kap.max()), 0.5 * (mu.min() + mu.max())))
    l0 = k0 - 2.0 / d * m0
    # wave vectors: real directions (G, G^C, G^R: k = phase * i * kr, the phase cancels) or complex (G^W)
    q, nyq = [], torch.zeros((1,) * d, dtype=torch.bool, device="cuda")
    for i in range(d):
        L = shape[d - 1 - i]
        m = torch.arange(L // 2 + 1 if i == 0 and not full else L, device="cuda", dtype=torch.float64)
        m = torch.where(m <= L // 2, m, m - L)
        view = [1] * d
        view[d - 1 - i] = -1
        q.append((2 * math.pi * m / L).view(view))
        if L % 2 == 0:
            nyq = nyq | (m == L // 2).view(view)
    clean = lambda t: torch.where(t.abs() < 1e-12, torch.zeros_like(t), t)  # sin(pi), cos(pi / 2)
    if green == "W":
        k = [torch.complex(clean(torch.cos(x)) - 1, clean(torch.sin(x))) for x in q]
    elif green == "MS":
        k = q
    elif green == "C":
        k = [clean(torch.sin(x)) for x in q]
    else:
        k = [2 * torch.sin(q[i] / 2) * math.prod(clean(torch.cos(q[j] / 2)) for j in range(d) if j != i)
             for i in range(d)]
    K2 = sum((x * x.conj()).real if green == "W" else x * x for x in k)
    zero = K2 == 0
    inv = torch.where(zero, torch.zeros_like(K2), 1.0 / torch.where(zero, torch.ones_like(K2), K2))
    if green == "W":
        A = torch.stack([torch.stack([l0 * k[j].conj() * k[l] + m0 * k[j] * k[l].conj()
                                      + (m0 * K2 + zero if j == l else torch.zeros_like(K2))
                                      for l in range(d)], -1) for j in range(d)], -2)
        Ainv = torch.linalg.inv(A)
        del A
    at = {ij: c for c, ij in enumerate(IJ)}
    comp = lambda i, j: at[(min(i, j), max(i, j))]
    w = torch.ones((), device="cuda", dtype=torch.float64)
    if not full:
        n1 = shape[-1]
        m = torch.arange(n1 // 2 + 1, device="cuda")
        w = torch.where((m == 0) | (2 * m == n1), 1.0, 2.0).double()
    fft = (lambda x: torch.fft.fftn(x, dim=tuple(a - 1 for a in axes))) if full else \
        (lambda x: torch.fft.rfftn(x, dim=tuple(a - 1 for a in axes)))
    ifft = (lambda x: torch.fft.ifftn(x, dim=tuple(a - 1 for a in axes)).real) if full else \
        (lambda x: torch.fft.irfftn(x, s=shape, dim=tuple(a - 1 for a in axes)))
    stress = lambda e: [(lf * sum(e[:d]) if c < d else 0.0) + 2 * mf * e[c] for c in range(len(IJ))]
    div = lambda s, j: sum((k[i].conj() if green == "W" else k[i]) * s[comp(i, j)] for i in range(d))
    eb = [float(eps_bar[i][j]) for i, j in IJ]
    two = [1.0 if c < d else 2.0 for c in range(len(IJ))]
    eps = [torch.full(shape, v, device="cuda", dtype=torch.float64) for v in eb]
    k_p, m_p = lf + 2.0 / d * mf, mf
    ak, am = (k0 / (k_p + k0), m0 / (m_p + m0)) if scheme == "AS" else (None, None)
    etas, means = [], []
    for it in range(max_iter):
        sig = stress(eps)
        ms, me = [float(s.mean()) for s in sig], [float(e.mean()) for e in eps]
        sh = [fft(s) for s in sig]
        num = sum(float((w * div(sh, j).abs().square()).sum()) for j in range(d))
        eta = math.sqrt(num) / (N * math.sqrt(sum(t * v * v for t, v in zip(two, ms))))
        etas.append(eta)
        means.append(ms)
        off = math.sqrt(sum(t * (a - b) ** 2 for t, a, b in zip(two, me, eb)) / sum(t * b * b for t, b in zip(two, eb)))
        if stop == "eta" and eta <= tol and (scheme == "DS" or off <= tol):
            break
        # tau_hat = sigma_hat - C0 : eps_hat, e = eps_bar - G' : tau
        trace = None
        for c in range(len(IJ)):
            eh = fft(eps[c])
            sh[c] -= 2 * m0 * eh
            if c < d:
                trace = eh if trace is None else trace + eh
        for c in range(d):
            sh[c] -= l0 * trace
        del trace, eh
        b = [div(sh, j) for j in range(d)]
        if green == "W":
            u = [sum(Ainv[..., j, l] * b[l] for l in range(d)) for j in range(d)]
        else:
            kb = sum(k[j] * b[j] for j in range(d)) * ((l0 + m0) / (l0 + 2 * m0)) * inv
            u = [(b[j] - k[j] * kb) * (inv / m0) for j in range(d)]
            del kb
        del b
        new = []
        for c, (i, j) in enumerate(IJ):
            h = -0.5 * (k[i] * u[j] + k[j] * u[i])
            if green == "MS":  # G = C0^-1 at the modes of eq. (hfreq)
                tr = sum(sh[a] for a in range(d))
                a2 = l0 / (2 * m0 * (d * l0 + 2 * m0))
                h = torch.where(nyq, -(sh[c] / (2 * m0) - (a2 * tr if c < d else 0.0)), h)
            else:
                h = torch.where(zero, torch.zeros_like(h), h)
            h.view(-1)[0] = eb[c] * N
            new.append(ifft(h))
        del sh, u, h
        if scheme == "AS":
            dl = [n - e for n, e in zip(new, eps)]
            tr = sum(dl[:d])
            new = [e + 2 * am * x + (2 * (ak - am) / d * tr if c < d else 0.0)
                   for c, (e, x) in enumerate(zip(eps, dl))]
            del dl, tr
        if stop == "maxdelta":
            change = max(float((a - b).abs().max()) for a, b in zip(new, eps))
            s2 = stress(new)
            change = max(change, max(float((a - b).abs().max()) for a, b in zip(s2, sig)))
            eps = new
            if change < tol:
                break
        else:
            eps = new
    sig = stress(eps)
    return (torch.stack(eps), torch.stack(sig), np.array([float(s.mean()) for s in sig]),
            np.array([float(e.mean()) for e in eps]), np.array(etas), np.array(means))


def _exact_net(phase, contrast, weights):
    """The network in 64 bits: periodic convolutions as sums of shifted matrix products."""
    def conv(name, x, skip=None, relu=True):
        wt, b = (torch.tensor(v, device="cuda").double() for v in weights[name])
        r = wt.shape[-1] // 2
        y = b.view(-1, 1, 1, 1).expand(-1, *x.shape[1:]).clone()
        for z in range(-r, r + 1):
            for v in range(-r, r + 1):
                for h in range(-r, r + 1):
                    xs = torch.roll(x, (-z, -v, -h), (1, 2, 3)).reshape(x.shape[0], -1)
                    y += (wt[:, :, z + r, v + r, h + r] @ xs).reshape(y.shape)
        if skip is not None:
            y += skip
        return y.clamp_min(0) if relu else y

    pool = lambda x: torch.nn.functional.avg_pool3d(x[None], 2)[0]
    up = lambda x: x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
    ind = (phase == 1).double()
    e0 = conv("enc0", torch.stack([ind, torch.full_like(ind, math.log10(contrast) - 2.0)]))
    e1 = conv("enc1b", conv("enc1a", pool(e0)))
    e2 = conv("enc2b", conv("enc2a", pool(e1)))
    e3 = conv("enc3b", conv("enc3a", pool(e2)))
    d2 = conv("dec2", up(e3), skip=e2)
    d1 = conv("dec1", up(d2), skip=e1)
    return conv("out", conv("dec0", up(d1), skip=e0), relu=False).reshape(-1)


def exact(case, seed):
    if case["kind"] == "warm":
        return _exact_net(_boolean(_shape(case), case["radius"], case["fraction"], seed), case["contrast"],
                          _weights(seed))
    if case["kind"] == "batched":
        return None  # over 20 seconds: two dozen solves of a hundred 64-bit iterations each
    phase = _boolean(_shape(case), case["radius"], case["fraction"], seed)
    lam, mu = _phases(case["contrast"])
    strain, stress, ms, me, eta, hist = _exact_solve(phase, lam, mu, _load(phase.ndim, seed), case["green"],
                                                     case["scheme"], case["tol"], case["max_iter"], case["stop"])
    if case["precision"] == "fp64":
        return dict(strain=strain, stress=stress, mean_stress=ms, mean_strain=me)
    out = dict(strain=strain, mean_stress=ms, mean_strain=me)
    if case["tol"] == 0.0:
        out["eta"], out["modulus"] = eta, hist
    return out
