"""The work that programs give this library, as cases that can be timed.

Each case is one public call, or the short sequence of calls that a program
makes for one result.  Its sizes are those of the tests and of bench.py:
images from 32^2 to 2048^2, 1000 to 200000 spiral samples, every precision,
penalty and minimiser, grids that are powers of two and grids that are not.

Solves run a few iterations, as in a dynamic series where every frame starts
from the one before it: the iteration costs the same whatever its number, and
after many iterations the rounding of any one sum decides the iterate (PR+
restarts), so that two correct results could not be compared.  The device
solves take no J history, which is optional there.

Data are the closed-form Fourier transforms of ellipses on spiral
trajectories, with complex Gaussian noise: what a scanner delivers, made
without any operator of the library.
"""
import math

import numpy as np
import torch

from paper_0908_3252_gb300 import spirec, synth

PRECISIONS = {"fp32": spirec.SPIREC_FP32, "fp16x3": spirec.SPIREC_MIXED_FP16X3, "bf16x3": spirec.SPIREC_MIXED_BF16X3}
PHIS = {"huber": spirec.SPIREC_PHI_HUBER, "hyperbolic": spirec.SPIREC_PHI_HYPERBOLIC,
        "quadratic": spirec.SPIREC_PHI_QUADRATIC}
MINIMISERS = {"half_quadratic": spirec.SPIREC_MIN_HALF_QUADRATIC, "newton": spirec.SPIREC_MIN_NEWTON}
# lambda1, alpha1, lambda0, alpha0 on images of intensity about 1
REG = {"huber": (0.05, 0.05, 0.02, 0.1), "hyperbolic": (0.2, 0.05, 0.05, 0.1), "quadratic": (0.5, 0.05, 0.2, 0.1)}
SERIES_INTERLEAVES, SERIES_SAMPLES, SERIES_SUBSET = 16, 2048, 4
SERIES_M = {128: 256, 192: 512, 256: 512}


def listed():
    return [
        # the normal operator inside a user's own solver, on a small image: launches and latency
        dict(name="toeplitz_64", op="toeplitz", N=64, arms=8, samples=1024, precision="fp32"),
        # simulating data of the 512^2 configuration
        dict(name="forward_512", op="forward", N=512, arms=32, samples=4096, precision="fp16x3"),
        # one coil's data brought to the image, sizes that divide no tile, the other 16-bit split
        dict(name="adjoint_250", op="adjoint", N=250, arms=15, samples=2111, precision="bf16x3"),
        # a new trajectory and its data, the 512^2 configuration: the operands of every later solve
        dict(name="setup_512", op="setup", N=512, arms=32, samples=4096, precision="fp16x3"),
        # the same at the 256^2 configuration, which asks for plain FP32
        dict(name="setup_256_fp32", op="setup", N=256, arms=16, samples=2048, precision="fp32"),
        # the image-domain solve at the paper's simulated size, starting from the previous frame
        dict(name="solve_128", op="solve", N=128, arms=6, samples=512, precision="fp16x3", phi="huber", iters=4,
             warm=True),
        # the 512^2 configuration's solve
        dict(name="solve_512", op="solve", N=512, arms=32, samples=4096, precision="fp16x3", phi="huber", iters=4,
             warm=False),
        # the largest size of the serving range, on the grid a plan picks for it by itself (768)
        dict(name="solve_384", op="solve", N=384, arms=16, samples=4096, precision="bf16x3", phi="hyperbolic",
             iters=4, warm=False),
        # the largest image, far beyond the L2
        dict(name="solve_2048", op="solve", N=2048, arms=64, samples=2048, precision="fp16x3", phi="huber", iters=4,
             warm=False),
        # truncated Newton, one of the two other minimisers
        dict(name="newton_256", op="outer", N=256, arms=16, samples=2048, precision="fp16x3", phi="hyperbolic",
             minimiser="newton", iters=2, inner=3),
        # a dynamic series: frames of three sizes, each from its own subset of cached interleaves
        dict(name="series_12", op="series", frames=12, precision="fp16x3", phi="huber", iters=4),
        # one request from host memory to host memory
        dict(name="host_192", op="host", N=192, arms=16, samples=1250, precision="fp16x3", phi="huber", iters=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _samples(rng, lo, hi):
    """arms x samples with a product spread over [lo, hi], most of them odd."""
    arms = rng.choice([3, 4, 6, 8, 11, 16, 24, 32])
    return dict(arms=arms, samples=max(2, _log_int(rng, lo, hi) // arms))


def draw(rng):
    op = rng.choice(["toeplitz", "forward", "adjoint", "setup", "solve", "solve", "outer", "series", "host"])
    if op == "toeplitz":
        return dict(op=op, N=_log_int(rng, 32, 1024), **_samples(rng, 1000, 65536),
                    precision=rng.choice(["fp32", "fp16x3"]))
    if op in ("forward", "adjoint", "setup"):
        precision = rng.choice(["fp32", "fp16x3", "bf16x3"])
        small = precision == "fp32"
        return dict(op=op, N=_log_int(rng, 32, 256 if small else 512),
                    **_samples(rng, 1000, 32768 if small else 131072), precision=precision)
    if op == "solve":
        return dict(op=op, N=_log_int(rng, 32, 768), **_samples(rng, 1000, 131072),
                    precision=rng.choice(["fp16x3", "bf16x3"]), phi=rng.choice(sorted(PHIS)),
                    iters=rng.randint(3, 4), warm=rng.random() < 0.5)
    if op == "outer":
        return dict(op=op, N=_log_int(rng, 32, 384), **_samples(rng, 1000, 65536),
                    precision=rng.choice(["fp16x3", "bf16x3"]), phi=rng.choice(["huber", "hyperbolic"]),
                    minimiser=rng.choice(sorted(MINIMISERS)), iters=rng.randint(1, 2), inner=rng.randint(3, 4))
    if op == "series":
        return dict(op=op, frames=rng.randint(3, 16), precision=rng.choice(["fp16x3", "bf16x3"]),
                    phi=rng.choice(["huber", "hyperbolic"]), iters=rng.randint(3, 4))
    return dict(op=op, N=_log_int(rng, 64, 384), **_samples(rng, 8000, 200000),
                precision=rng.choice(["fp16x3", "bf16x3"]), phi=rng.choice(["huber", "hyperbolic"]),
                iters=rng.randint(3, 4))


# ------------------------------------------------------------------- inputs


class _Object:
    """Ten ellipses with complex intensities: rasterised, or transformed."""

    def __init__(self, N, g):
        u = g.uniform
        self.N = N
        self.c = (N - 1) / 2.0 + u(-0.35, 0.35, (10, 2)) * N
        self.ab = u(0.05, 0.3, (10, 2)) * N
        self.th = u(0.0, np.pi, 10)
        self.amp = u(0.0, 1.0, 10) * np.exp(1j * u(-0.5, 0.5, 10))

    def image(self, shift=0.0):
        n = torch.arange(self.N, dtype=torch.float64, device="cuda")
        out = torch.zeros((self.N, self.N), dtype=torch.complex128, device="cuda")
        for (cx, cy), (a, b), th, amp in zip(self.c + shift, self.ab, self.th, self.amp):
            y, x = (n - cy)[:, None], (n - cx)[None, :]
            xr, yr = x * math.cos(th) + y * math.sin(th), y * math.cos(th) - x * math.sin(th)
            out += complex(amp) * (((xr / a) ** 2 + (yr / b) ** 2) <= 1.0)
        return out

    def samples(self, kx, ky):
        out = torch.zeros(kx.shape[0], dtype=torch.complex128, device="cuda")
        for (cx, cy), (a, b), th, amp in zip(self.c, self.ab, self.th, self.amp):
            kr = a * (kx * math.cos(th) + ky * math.sin(th))
            ki = b * (ky * math.cos(th) - kx * math.sin(th))
            rho = torch.sqrt(kr * kr + ki * ki).clamp_min(1e-9)
            out += complex(amp) * a * b * torch.special.bessel_j1(2.0 * math.pi * rho) / rho * _cis(kx * cx + ky * cy)
        return out / self.N


def _cis(turns):
    a = 2.0 * math.pi * (turns - torch.round(turns))
    return torch.complex(torch.cos(a), torch.sin(a))


def _noise(shape, gen):
    return torch.complex(*(torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2)))


def _spiral(N, arms, samples, rotation, kind="archimedean", arm_rotation="uniform"):
    kx, ky = synth.spiral(N, arms, samples, kind, arm_rotation)
    c, s = math.cos(rotation), math.sin(rotation)
    return (torch.from_numpy(np.clip(c * kx - s * ky, -0.5, 0.5)).cuda(),
            torch.from_numpy(np.clip(s * kx + c * ky, -0.5, 0.5)).cuda())


def _data(obj, kx, ky, gen):
    """30 dB data of the object."""
    s = obj.samples(kx, ky)
    return (s + s.abs().square().mean().sqrt() * 10 ** -1.5 / math.sqrt(2.0) * _noise(s.shape, gen)).to(torch.complex64)


def _inputs(case, seed):
    g, gen = np.random.default_rng(seed), torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rotation = g.uniform(0.0, 2.0 * np.pi)
    if case["op"] == "series":
        kx, ky = _spiral(256, SERIES_INTERLEAVES, SERIES_SAMPLES, rotation, "archimedean", "golden")
        frames = []
        for i in range(case["frames"]):
            N = sorted(SERIES_M)[i % len(SERIES_M)]
            which = np.sort(g.choice(SERIES_INTERLEAVES, SERIES_SUBSET, replace=False)).astype(np.int32)
            arm = torch.arange(SERIES_SAMPLES, device="cuda")
            at = torch.cat([arm + int(j) * SERIES_SAMPLES for j in which])
            obj = _Object(N, g)
            frames.append(dict(N=N, which=which, kx=kx[at], ky=ky[at], s=_data(obj, kx[at], ky[at], gen)))
        return dict(kx=kx, ky=ky, frames=frames)
    N = case["N"]
    kx, ky = _spiral(N, case["arms"], case["samples"], rotation)
    obj = _Object(N, g)
    out = dict(kx=kx, ky=ky, s=_data(obj, kx, ky, gen))
    if case["op"] in ("toeplitz", "forward"):
        out["x"] = (obj.image() + 0.05 * _noise((N, N), gen)).to(torch.complex64)
    if case.get("warm"):
        # the previous frame: the same object a little elsewhere, with its own noise
        out["x0"] = (obj.image(0.7) + 0.03 * _noise((N, N), gen)).to(torch.complex64)
    return out


class _Caches:
    """The per-interleave kernel caches of a series, one per image size."""

    def __init__(self, sizes, kx, ky, precision):
        offsets = np.arange(SERIES_INTERLEAVES + 1) * SERIES_SAMPLES
        self.h = {N: spirec.spirec_kcache_create(N, SERIES_M[N], precision, offsets, kx.cpu().numpy(),
                                                 ky.cpu().numpy()) for N in sizes}

    def __del__(self):
        for h in self.h.values():
            spirec.spirec_kcache_destroy(h)


def _plan(N, L, precision, M=0, phi=None):
    p = spirec.Plan(N, L, M, precision, torch.cuda.current_stream().cuda_stream)
    if phi is not None:
        spirec.spirec_set_reg(p.h, *REG[phi], PHIS[phi])
    return p


def prepare(case, seed):
    op, precision, d = case["op"], PRECISIONS[case["precision"]], _inputs(case, seed)
    st = dict(case=case)
    if op == "series":
        st["caches"] = _Caches({f["N"] for f in d["frames"]}, d["kx"], d["ky"], precision)
        st["frames"] = []
        for f in d["frames"]:
            p = _plan(f["N"], f["s"].shape[0], precision, SERIES_M[f["N"]], case["phi"])
            x = torch.empty((f["N"], f["N"]), dtype=torch.complex64, device="cuda")
            st["frames"].append((p, st["caches"].h[f["N"]], f["which"], f["s"], x))
        return st
    N, L = case["N"], d["s"].shape[0]
    p = st["plan"] = _plan(N, L, precision, phi=case.get("phi"))
    if op == "host":
        st["kx"], st["ky"], st["s"] = (d[k].cpu().numpy() for k in ("kx", "ky", "s"))
        return st
    image = lambda: torch.empty((N, N), dtype=torch.complex64, device="cuda")  # noqa: E731
    if op == "setup":
        st.update(kx=d["kx"], ky=d["ky"], s=d["s"], D=image(),
                  C=torch.empty((p.M, p.M), dtype=torch.float32, device="cuda"))
        return st
    spirec.spirec_set_trajectory_dev(p.h, d["kx"], d["ky"])
    if op == "toeplitz":
        st.update(x=d["x"], Tx=image())
    elif op == "forward":
        st.update(x=d["x"], y=torch.empty(L, dtype=torch.complex64, device="cuda"))
    elif op == "adjoint":
        st.update(y=d["s"], x=image())
    else:
        if op == "outer":
            spirec.spirec_set_minimiser(p.h, MINIMISERS[case["minimiser"]], case["inner"])
        spirec.spirec_set_data_dev(p.h, d["s"])
        st.update(x0=d.get("x0"), x=image())
    spirec.spirec_sync(p.h)
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "series":
        for p, cache, which, s, x in st["frames"]:
            spirec.spirec_set_trajectory_cached(p.h, cache, which)
            spirec.spirec_set_data_dev(p.h, s)
        spirec.spirec_batch_solve([f[0].h for f in st["frames"]], [f[4] for f in st["frames"]], case["iters"])
        return [f[4] for f in st["frames"]]
    p = st["plan"]
    if op == "toeplitz":
        spirec.spirec_toeplitz_dev(p.h, st["x"], st["Tx"])
        return st["Tx"]
    if op == "forward":
        spirec.spirec_forward_dev(p.h, st["x"], st["y"])
        return st["y"]
    if op == "adjoint":
        spirec.spirec_adjoint_dev(p.h, st["y"], st["x"])
        return st["x"]
    if op == "setup":
        spirec.spirec_set_trajectory_dev(p.h, st["kx"], st["ky"])
        spirec.spirec_set_data_dev(p.h, st["s"])
        spirec.spirec_kernel_spectrum_dev(p.h, st["C"])
        spirec.spirec_data_adjoint_dev(p.h, st["D"])
        return [st["C"], st["D"]]
    if op == "host":
        spirec.spirec_set_trajectory(p.h, st["kx"], st["ky"])
        spirec.spirec_set_data(p.h, st["s"])
        # the J history comes with the host call; it is a report in 64 bits of sums in 32 that cancel to
        # 1e-4 of their terms, and the image is the result
        return spirec.spirec_solve(p.h, None, case["iters"], p.N)[0]
    spirec.spirec_solve_dev(p.h, st["x0"], case["iters"], st["x"], None)
    return st["x"]


# --------------------------------------------------------------------- work


def _grid(N):
    """The grid that a plan picks: the smallest 2^a 3^b 5^c >= 2N - 1."""
    M = 2 * N - 1
    while True:
        r = M
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1:
            return M
        M += 1


def _apply_flops(N, M):
    """N row FFTs and M column FFTs there and back, and the spectrum."""
    return 2.0 * (N + M) * 5.0 * M * math.log2(M) + 2.0 * M * M


def work(case):
    op = case["op"]
    if op == "series":
        total = dict(bytes=0.0, flops=0.0)
        L = SERIES_SUBSET * SERIES_SAMPLES
        for i in range(case["frames"]):
            N = sorted(SERIES_M)[i % len(SERIES_M)]
            M = SERIES_M[N]
            total["bytes"] += SERIES_SUBSET * (4.0 * M * M + 8.0 * N * (2 * N - 1)) + 24.0 * L + 8.0 * N * N
            total["flops"] += 8.0 * N * N * L + case["iters"] * (_apply_flops(N, M) + 100.0 * N * N)
        return total
    N, L = case["N"], case["arms"] * case["samples"]
    M = _grid(N)
    nudft, gram, image = 8.0 * N * N * L, 8.0 * N * (2 * N - 1) * L, 8.0 * N * N
    if op == "toeplitz":
        return dict(bytes=2 * image + 4.0 * M * M, flops=_apply_flops(N, M))
    if op in ("forward", "adjoint"):
        return dict(bytes=image + 24.0 * L, flops=nudft)
    if op == "setup":
        return dict(bytes=24.0 * L + image + 4.0 * M * M, flops=nudft + gram)
    applies = case["iters"] * case.get("inner", 1)
    solve = dict(bytes=3 * image + 4.0 * M * M, flops=applies * (_apply_flops(N, M) + 100.0 * N * N))
    if op == "host":
        return dict(bytes=24.0 * L + image, flops=solve["flops"] + nudft + gram)
    return solve


# -------------------------------------------------- the same in 64 bits


def _phases(k, n, chunk):
    """exp(i 2 pi k_l j), j < n, for a chunk of samples."""
    return _cis(k[chunk, None] * torch.arange(n, dtype=torch.float64, device="cuda"))


def _chunks(L, n):
    step = max(1, (1 << 25) // n)
    return [slice(i, min(L, i + step)) for i in range(0, L, step)]


def _forward64(kx, ky, f):
    N = f.shape[0]
    return torch.cat([((_phases(kx, N, c) @ f.T) * _phases(ky, N, c)).sum(1) for c in _chunks(kx.shape[0], N)]) / N


def _adjoint64(kx, ky, s, N):
    out = torch.zeros((N, N), dtype=torch.complex128, device="cuda")
    for c in _chunks(kx.shape[0], N):
        out += (_phases(ky, N, c).conj() * s[c, None]).T @ _phases(kx, N, c).conj()
    return out / N


def _spectrum64(kx, ky, N, M):
    """The DFT of the circulant that holds conj G, over M^2: real."""
    G = torch.zeros((2 * N - 1, N), dtype=torch.complex128, device="cuda")  # [v + N - 1, u]
    for c in _chunks(kx.shape[0], 2 * N):
        e = _phases(ky, 2 * N - 1, c) * _cis(-ky[c, None] * (N - 1))
        G += e.T @ _phases(kx, N, c)
    G /= N * N
    full = torch.cat([torch.flip(G[:, 1:], (0, 1)).conj(), G], 1)  # G at -u, -v is conj G
    at = torch.arange(-(N - 1), N, device="cuda") % M
    c = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
    c[at[:, None], at[None, :]] = full.conj()
    return torch.fft.fft2(c).real / (M * M)


def _apply64(C, x):
    N, M = x.shape[0], C.shape[0]
    return torch.fft.ifft2(torch.fft.fft2(x, s=(M, M)) * C)[:N, :N] * (M * M)


def _dot(a, b):
    return float((a.real * b.real + a.imag * b.imag).sum())


def _right(x):
    return x[:, 1:] - x[:, :-1]


def _down(x):
    return x[1:] - x[:-1]


def _back(terms):
    """The adjoint of (right differences, down differences, pixels)."""
    r, d, p = terms
    out = p.clone()
    out[:, 1:] += r
    out[:, :-1] -= r
    out[1:] += d
    out[:-1] -= d
    return out


class _Penalty:
    def __init__(self, phi):
        self.phi = phi
        l1, a1, l0, a0 = (float(np.float32(v)) for v in REG[phi])  # the library keeps them in FP32
        self.la = ((l1, a1), (l1, a1), (l0, a0))

    def terms(self, x):
        return (_right(x), _down(x), x)

    def weight(self, alpha, r):
        """phi'(r) / r"""
        if self.phi == "huber":
            return torch.where(r <= alpha, 2.0, 2.0 * alpha / r.clamp_min(1e-300))
        if self.phi == "hyperbolic":
            return 2.0 * alpha / torch.sqrt(alpha * alpha + r * r)
        return torch.full_like(r, 2.0)

    def bend(self, alpha, r):
        """(phi''(r) - phi'(r) / r) / r^2"""
        if self.phi == "huber":
            return torch.where(r <= alpha, 0.0, -2.0 * alpha / r.clamp_min(alpha) ** 3)
        if self.phi == "hyperbolic":
            return -2.0 * alpha / (alpha * alpha + r * r) ** 1.5
        return torch.zeros_like(r)

    def grad(self, x):
        return _back([lam * self.weight(a, z.abs()) * z for (lam, a), z in zip(self.la, self.terms(x))])

    def line(self, f, d, t):
        num = den = 0.0
        for (lam, a), z, w in zip(self.la, self.terms(f), self.terms(d)):
            z = z + t * w
            b = lam * self.weight(a, z.abs())
            num += _dot(b * z, w)
            den += _dot(b * w, w)
        return num, den

    def weighted(self, f):
        """x -> sum_e W_e delta_e^T delta_e x, W = lambda phi'(r) / (2 r) at f."""
        W = [0.5 * lam * self.weight(a, z.abs()) for (lam, a), z in zip(self.la, self.terms(f))]
        return lambda x: _back([w * t for w, t in zip(W, self.terms(x))])

    def half_hessian(self, f):
        z = self.terms(f)
        W = [0.5 * lam * self.weight(a, q.abs()) for (lam, a), q in zip(self.la, z)]
        E = [0.5 * lam * self.bend(a, q.abs()) for (lam, a), q in zip(self.la, z)]

        def apply(x):
            return _back([w * t + e * q * (q.real * t.real + q.imag * t.imag)
                          for w, e, q, t in zip(W, E, z, self.terms(x))])
        return apply


def _step64(pen, f, d, q1, q2):
    t = 0.0
    for _ in range(3):
        num, den = pen.line(f, d, t)
        if den + 2.0 * q2 > 0.0:
            t -= (num + q1 + 2.0 * q2 * t) / (den + 2.0 * q2)
    return t


def _prcg64(C, D, pen, f, iters):
    res = _apply64(C, f) - D
    g = 2.0 * res + pen.grad(f)
    d = -g
    for _ in range(iters):
        Td = _apply64(C, d)
        t = _step64(pen, f, d, 2.0 * _dot(d, res), _dot(d, Td))
        f, res = f + t * d, res + t * Td
        gn = 2.0 * res + pen.grad(f)
        gg = _dot(g, g)
        beta = max(0.0, _dot(gn, gn - g) / gg) if gg > 0.0 else 0.0
        d = -gn + beta * d
        if _dot(gn, d) >= 0.0:
            d = -gn
        g = gn
    return f


def _linear_cg64(A, x, r, steps):
    p, rho = r.clone(), _dot(r, r)
    for _ in range(steps):
        q = A(p)
        pq = _dot(p, q)
        a = rho / pq if pq > 0.0 else 0.0
        x, r = x + a * p, r - a * q
        new = _dot(r, r)
        p, rho = r + (new / rho if rho > 0.0 else 0.0) * p, new
    return x


def _outer64(C, D, pen, f, kind, outer, inner):
    for _ in range(outer):
        res = _apply64(C, f) - D
        if kind == "half_quadratic":
            P = pen.weighted(f)
            f = _linear_cg64(lambda x: _apply64(C, x) + P(x), f, -res - P(f), inner)
        else:
            P = pen.half_hessian(f)
            s = _linear_cg64(lambda x: _apply64(C, x) + P(x), torch.zeros_like(f), -res - 0.5 * pen.grad(f), inner)
            f = f + _step64(pen, f, s, 2.0 * _dot(s, res), _dot(s, _apply64(C, s))) * s
    return f


def exact(case, seed):
    op, d = case["op"], _inputs(case, seed)
    wide = lambda v: v.to(torch.complex128)  # noqa: E731
    if op == "series":
        out, pen = [], _Penalty(case["phi"])
        for f in d["frames"]:
            N = f["N"]
            C = _spectrum64(f["kx"], f["ky"], N, SERIES_M[N])
            D = _adjoint64(f["kx"], f["ky"], wide(f["s"]), N)
            out.append(_prcg64(C, D, pen, torch.zeros_like(D), case["iters"]))
        return out
    N, kx, ky = case["N"], d["kx"], d["ky"]
    if op == "forward":
        return _forward64(kx, ky, wide(d["x"]))
    if op == "adjoint":
        return _adjoint64(kx, ky, wide(d["s"]), N)
    C = _spectrum64(kx, ky, N, _grid(N))
    if op == "toeplitz":
        return _apply64(C, wide(d["x"]))
    D = _adjoint64(kx, ky, wide(d["s"]), N)
    if op == "setup":
        return [C, D]
    pen = _Penalty(case["phi"])
    f = wide(d["x0"]) if "x0" in d else torch.zeros_like(D)
    if op == "outer":
        f = _outer64(C, D, pen, f, case["minimiser"], case["iters"], case["inner"])
    else:
        f = _prcg64(C, D, pen, f, case["iters"])
    return f.cpu().numpy() if op == "host" else f
