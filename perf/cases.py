"""The work that users of the BdG library have it do, as timed cases.

Each case is one call of a public entry point of paper_2506_08308_gb300.bdg on
the problems the repository is used for: the 1-D, 2-D and 3-D workloads of
synth.py (grids, boxes, interaction constants, block sizes), the batched
workload's parameter ranges, and the paper's perturbed densities.

  apply    y = M x, the block product (both forms, both precisions, 1-D to 3-D)
  gram     the Gram contraction of two column blocks (both engines)
  biortho  bi-orthonormalisation against a locked pair
  density  perturbed densities of excitation modes
  ground   the ground state, host arrays in and out
  solve    the k smallest excitation energies
"""
import functools
import math

import numpy as np
import torch

from paper_2506_08308_gb300 import bdg

FORM = {"uv": bdg.UV, "fg": bdg.FG}
CPLX = {"c64": torch.complex64, "c128": torch.complex128}
REAL = {"c64": torch.float32, "c128": torch.float64}
ENGINE = {"simt": bdg.GRAM_SIMT, "tensor": bdg.GRAM_TENSOR}
PREC = {"fp64": bdg.FP64, "mixed": bdg.MIXED}


# ------------------------------------------------------------------- cases
def listed():
    p1 = {"nx": 256, "ny": 0, "nz": 0, "box": 16.0, "gy": 1.0, "gz": 1.0, "beta_n": 10.0, "beta_s": -1.0,
          "p": 0.0, "q": 0.0}
    p2 = {"nx": 256, "ny": 256, "nz": 0, "box": 12.0, "gy": 1.0, "gz": 1.0, "beta_n": 100.0, "beta_s": -2.0,
          "p": 0.0, "q": 0.1}
    p3 = {"nx": 128, "ny": 128, "nz": 128, "box": 8.0, "gy": 1.5, "gz": 2.0, "beta_n": 200.0, "beta_s": -4.0,
          "p": 0.05, "q": 0.2}
    return [
        # the 1-D FP64 workload's block product: one launch on L2-resident data, latency counts
        {"name": "apply_1d_c128", "do": "apply", **p1, "dtype": "c128", "form": "fg", "nvec": 24},
        # a few amplitudes on a coarse rectangular grid (a check of a mode, a scan over parameters)
        {"name": "apply_2d_c64_small", "do": "apply", **p2, "nx": 64, "ny": 128, "dtype": "c64", "form": "uv", "nvec": 5},
        # the benchmark's FP32 block product, the bulk of the mixed solver's inner iterations
        {"name": "apply_2d_c64", "do": "apply", **p2, "dtype": "c64", "form": "fg", "nvec": 48},
        # FP64 residuals of the benchmark's 32 computed amplitudes (UV form)
        {"name": "apply_2d_c128", "do": "apply", **p2, "dtype": "c128", "form": "uv", "nvec": 32},
        # the 3-D workload's FP32 block product, the largest arrays
        {"name": "apply_3d_c64", "do": "apply", **p3, "dtype": "c64", "form": "fg", "nvec": 48},
        # Gram-Schmidt coefficients of one block of 24 pair columns against another (256^2, three components)
        {"name": "gram_tensor_c128", "do": "gram", "engine": "tensor", "dtype": "c128", "ca": 24, "cb": 24, "n": 3 * 65536},
        # projected matrix of the Rayleigh-Ritz step on three blocks, FP64 accuracy
        {"name": "gram_simt_c128", "do": "gram", "engine": "simt", "dtype": "c128", "ca": 72, "cb": 72, "n": 3 * 65536},
        # a new block of 24 columns made bi-orthonormal against 24 locked pairs, middle grid of the batched workload
        {"name": "biortho_c128", "do": "biortho", **p2, "nx": 128, "ny": 128, "dtype": "c128", "ncol": 24, "nlock": 24},
        # density figures: 32 modes of the 256^2 workload at one time
        {"name": "density_c64", "do": "density", **p2, "dtype": "c64", "nmode": 32, "nt": 1},
        # ground state of a coarse 2-D instance, as every solve begins with one
        {"name": "ground_2d", "do": "ground", **p2, "nx": 64, "ny": 64},
        # whole FP64 solve of the 1-D workload
        {"name": "solve_1d_fp64", "do": "solve", **p1, "prec": "fp64", "k": 16, "m": 24},
        # whole mixed-precision solve of the 2-D benchmark instance
        {"name": "solve_2d_mixed", "do": "solve", **p2, "prec": "mixed", "k": 32, "m": 48},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def _physics(rng, nx, ny, nz):
    two = {"box": 12.0, "beta_n": rng.uniform(50.0, 200.0), "beta_s": rng.uniform(-5.0, 5.0), "p": 0.0,
           "q": rng.uniform(0.05, 0.5)}
    one = {"box": 16.0, "beta_n": rng.uniform(5.0, 20.0), "beta_s": rng.uniform(-2.0, -0.5), "p": 0.0, "q": 0.0}
    three = {"box": 8.0, "beta_n": rng.uniform(100.0, 400.0), "beta_s": rng.uniform(-8.0, 5.0), "p": 0.05, "q": 0.2}
    return {"nx": nx, "ny": ny, "nz": nz, "gy": 1.0, "gz": 1.0, **(three if nz else two if ny else one)}


def draw(rng):
    do = rng.choice(["apply", "apply", "apply", "gram", "gram", "biortho", "density", "ground", "solve"])
    dtype = rng.choice(["c64", "c128"])
    if do == "apply":
        dim = rng.choice([1, 2, 2, 3])
        n = ([_pow2(rng, 64, 1024), 0, 0] if dim == 1 else [_pow2(rng, 32, 512), _pow2(rng, 32, 512), 0] if dim == 2
             else [_pow2(rng, 16, 128), _pow2(rng, 16, 128), _pow2(rng, 16, 128)])
        pts = math.prod(v for v in n if v)
        most = max(1, min(64, (48 * 65536 if dtype == "c128" else 24 * 2097152) // pts))
        return {"do": do, **_physics(rng, *n), "dtype": dtype, "form": rng.choice(["uv", "fg"]),
                "nvec": _log_int(rng, 1, most)}
    if do == "gram":
        return {"do": do, "engine": rng.choice(["simt", "tensor"]), "dtype": dtype, "ca": _log_int(rng, 2, 76),
                "cb": _log_int(rng, 2, 76), "n": _log_int(rng, 500, 400000)}
    if do == "biortho":
        n = rng.choice([[256, 0, 0], [64, 64, 0], [128, 64, 0], [128, 128, 0]])
        return {"do": do, **_physics(rng, *n), "dtype": dtype, "ncol": rng.randint(2, 40), "nlock": rng.randint(0, 60)}
    if do == "density":
        n = [_pow2(rng, 32, 256), _pow2(rng, 32, 256), 0]
        return {"do": do, **_physics(rng, *n), "dtype": dtype, "nmode": _log_int(rng, 1, 40), "nt": _log_int(rng, 1, 24)}
    if do == "ground":
        n = rng.choice([[128, 0, 0], [256, 0, 0], [64, 64, 0]])
        return {"do": do, **_physics(rng, *n)}
    k = rng.randint(6, 16)
    if rng.random() < 0.5:
        return {"do": do, **_physics(rng, rng.choice([128, 256]), 0, 0), "prec": rng.choice(["fp64", "mixed"]),
                "k": k, "m": k + 8}
    n = rng.choice([64, 128])
    return {"do": do, **_physics(rng, n, n, 0), "prec": "mixed", "k": k, "m": k + 8}


# ------------------------------------------------------------------ inputs
def _grid(c):
    return [c[a] for a in ("nx", "ny", "nz") if c[a]]


def _axes(c):
    return [-c["box"] + np.arange(n) * (2.0 * c["box"] / n) for n in _grid(c)]


def _potential(c):
    """Harmonic trap and the Gaussian of its lowest state."""
    V, r2 = 0.0, 0.0
    for x, g in zip(np.meshgrid(*_axes(c), indexing="ij"), (1.0, c["gy"], c["gz"])):
        V = V + 0.5 * (g * x) ** 2
        r2 = r2 + g * x * x
    return V, np.exp(-0.5 * r2)


def _params(c, **kw):
    n = _grid(c)
    return bdg.make_params(n, [-c["box"]] * len(n), [c["box"]] * len(n), c["beta_n"], c["beta_s"], c["p"], c["q"], **kw)


def _cell(c):
    return math.prod(2.0 * c["box"] / n for n in _grid(c))


def _spinor(c, seed):
    """A smooth real spinor of mass 1: a broad condensate, all components occupied."""
    rng = np.random.default_rng(seed)
    env = _potential(c)[1] ** 0.2
    phi = np.stack([w * env for w in 0.5 + rng.uniform(0.0, 1.0, 3)])
    return phi / math.sqrt(_cell(c) * float((phi * phi).sum()))


@functools.lru_cache(maxsize=8)
def _ground(items):
    """The ground state a solve starts from, found once per problem."""
    c = dict(items)
    V, env = _potential(c)
    phi0 = np.stack([w * env for w in 0.5 + np.random.default_rng(7).uniform(0.0, 1.0, 3)])
    return V, bdg.ground_state(_params(c), 0.0, V, phi0)[0]


def _problem(c):
    return tuple((a, c[a]) for a in ("nx", "ny", "nz", "box", "gy", "gz", "beta_n", "beta_s", "p", "q"))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(shape, dtype, g):
    return torch.randn(shape, dtype=CPLX[dtype], device="cuda", generator=g)


def _envelope(c, dtype):
    return torch.from_numpy(_potential(c)[1] ** 0.1).to("cuda", REAL[dtype]).reshape(-1)


def _columns(n, cols, dtype, g):
    """Columns of amplitudes that fall off towards the edges of the trap."""
    r = torch.linspace(-3.0, 3.0, n, device="cuda", dtype=REAL[dtype])
    return _normal((cols, n), dtype, g) * torch.exp(-0.5 * r * r)


def prepare(case, seed):
    c, g, do = case, _gen(seed), case["do"]
    if do == "apply":
        # the seeded complex Gaussian block every iteration starts from
        plan = bdg.Plan(_params(c), _potential(c)[0], _spinor(c, seed))
        return {"do": do, "plan": plan, "form": FORM[c["form"]], "x": _normal((c["nvec"], 6, plan.npts), c["dtype"], g)}
    if do == "gram":
        A, B = _columns(c["n"], c["ca"], c["dtype"], g), _columns(c["n"], c["cb"], c["dtype"], g)
        w = min(c["ca"], c["cb"])
        B[:w] = 0.5 * B[:w] + A[:w]     # neighbouring blocks of an iteration: the diagonal stands out
        return {"do": do, "A": A, "B": B, "engine": ENGINE[c["engine"]]}
    if do == "biortho":
        # Amplitudes of a real condensate are real: zero imaginary parts, as the solver returns them.
        plan = bdg.Plan(_params(c), _potential(c)[0], _spinor(c, seed))
        rdt, n3, k = REAL[c["dtype"]], 3 * plan.npts, c["ncol"] + c["nlock"]
        env = _envelope(c, "c128").repeat(3)
        q = torch.linalg.qr((torch.randn((k, n3), dtype=torch.float64, device="cuda", generator=g) * env).T)[0].T
        t = 0.5 + torch.rand((k, 1), dtype=torch.float64, device="cuda", generator=g)
        s = (1.0 + 0.15 * torch.arange(k, dtype=torch.float64, device="cuda"))[:, None]
        noise = 0.02 / math.sqrt(n3) * torch.randn((k, n3), dtype=torch.float64, device="cuda", generator=g)
        cols = lambda v: v.to(rdt).to(CPLX[c["dtype"]]).reshape(-1, 3, plan.npts).contiguous()  # noqa: E731
        lock = c["nlock"]
        F, G = q[lock:] * t[lock:], (q[lock:] * s[: c["ncol"]] / t[lock:] + noise[lock:])
        F, G = F + 0.1 * q[:lock].sum(0), G - 0.1 * q[:lock].sum(0)   # what the locked pairs take out
        return {"do": do, "plan": plan, "F": cols(F), "G": cols(G),
                "Fl": cols(q[:lock] * t[:lock]) if lock else None, "Gl": cols(q[:lock] / t[:lock]) if lock else None}
    if do == "density":
        plan = bdg.Plan(_params(c), _potential(c)[0], _spinor(c, seed))
        UV = _normal((c["nmode"], 6, plan.npts), c["dtype"], g) * _envelope(c, c["dtype"])
        rng = np.random.default_rng(seed)
        return {"do": do, "plan": plan, "UV": UV, "omega": rng.uniform(0.1, 3.0, c["nmode"]),
                "times": rng.uniform(0.0, 10.6, c["nt"])}
    if do == "ground":
        V, env = _potential(c)
        rng = np.random.default_rng(seed)
        phi0 = np.stack([w * env for w in 0.5 + rng.uniform(0.0, 1.0, 3)])
        return {"do": do, "prm": _params(c), "V": V, "phi0": phi0 * (1.0 + 0.05 * rng.standard_normal(phi0.shape))}
    V, phi = _ground(_problem(c))
    plan = bdg.Plan(_params(c, prec=PREC[c["prec"]], tol=1e-10, maxit=300), V, phi)
    return {"do": do, "plan": plan, "k": c["k"], "m": c["m"], "x": _normal((c["m"], 6, plan.npts), "c128", g)}


# --------------------------------------------------------------- the calls
def run(state):
    s, do = state, state["do"]
    if do == "apply":
        return s["plan"].apply(s["x"], s["form"])
    if do == "gram":
        return bdg.gram(s["A"], s["B"], s["engine"])
    if do == "biortho":
        # it works in place; the caller keeps the raw block
        F, G = s["F"].clone(), s["G"].clone()
        return {"rank": s["plan"].biortho(F, G, s["Fl"], s["Gl"]), "F": F, "G": G}
    if do == "density":
        return s["plan"].perturbed_density(s["UV"], s["omega"], s["times"], 0.1)
    if do == "ground":
        phi, mu = bdg.ground_state(s["prm"], 0.0, s["V"], s["phi0"])[:2]
        return {"phi": phi, "mu": mu}
    # the spectrum: vectors of degenerate pairs are any basis of theirs, residuals below the target are rounding
    omega, _, _, nconv = s["plan"].solve(s["k"], s["m"], X0=s["x"], want_vectors=False, allow_not_converged=True)
    return {"omega": omega, "nconv": nconv}


def work(case):
    c, do = case, case["do"]
    e = 8 if c.get("dtype") == "c64" else 16
    if do == "gram":
        return {"bytes": e * c["n"] * (c["ca"] + c["cb"]) + 32 * c["ca"] * c["cb"], "flops": 8 * c["n"] * c["ca"] * c["cb"]}
    pts = math.prod(_grid(c))
    # line FFTs forward and back along every axis, the multiplier, the pointwise 6 x 6 coupling
    product = 6 * pts * (sum(10 * math.log2(n) + 2 for n in _grid(c)) + 24)
    if do == "apply":
        return {"bytes": 12 * e * pts * c["nvec"] + 2 * e * pts, "flops": product * c["nvec"]}
    if do == "biortho":
        k, lock = c["ncol"], c["nlock"]
        return {"bytes": e * 3 * pts * (4 * k + 2 * lock), "flops": 8 * 3 * pts * (8 * k * lock + 3 * k * k)}
    if do == "density":
        return {"bytes": pts * (c["nmode"] * (6 * e + 1.5 * e * c["nt"]) + 2 * e),
                "flops": 3 * pts * c["nmode"] * (4 + 10 * c["nt"])}
    if do == "ground":
        return {"bytes": 8 * 7 * pts, "flops": product}
    # the start block and one evaluation of the residuals of k pairs
    return {"bytes": 96 * pts * c["m"], "flops": product * c["k"]}


# ------------------------------------------------------- the same in 64 bits
def _blocks(c, phi):
    """Pointwise A and B of the operator at a real spinor, without the chemical potentials' diagonal."""
    a, b, m = phi
    V, bn, bs = _potential(c)[0].reshape(-1), c["beta_n"], c["beta_s"]
    rho = a * a + b * b + m * m
    A = np.empty((3, 3, a.size))
    A[0, 0] = V + c["q"] - c["p"] + bn * (rho + a * a) + bs * (2 * a * a + b * b - m * m)
    A[1, 1] = V + bn * (rho + b * b) + bs * (a * a + m * m)
    A[2, 2] = V + c["q"] + c["p"] + bn * (rho + m * m) + bs * (2 * m * m + b * b - a * a)
    A[0, 1] = A[1, 0] = bn * a * b + bs * b * (a + 2 * m)
    A[1, 2] = A[2, 1] = bn * b * m + bs * b * (2 * a + m)
    A[0, 2] = A[2, 0] = (bn - bs) * a * m
    B = np.empty_like(A)
    B[0, 0], B[1, 1], B[2, 2] = (bn + bs) * a * a, bn * b * b + 2 * bs * a * m, (bn + bs) * m * m
    B[0, 1] = B[1, 0] = (bn + bs) * a * b
    B[1, 2] = B[2, 1] = (bn + bs) * b * m
    B[0, 2] = B[2, 0] = bn * a * m + bs * (b * b - a * m)
    return A, B


def _symbol(c):
    k2 = 0.0
    for n in np.meshgrid(*[2 * np.pi * np.fft.fftfreq(n, 2.0 * c["box"] / n) for n in _grid(c)], indexing="ij"):
        k2 = k2 + 0.5 * n * n
    return k2


def _minus_mu(c, phi, A, B):
    """A less the chemical potentials mu_j = <phi_j, (H phi)_j> / |phi_j|^2, with H = (A - B) and the kinetic part."""
    n, ax = _grid(c), tuple(range(1, 1 + len(_grid(c))))
    h = np.fft.ifftn(_symbol(c) * np.fft.fftn(phi.reshape([3] + n), axes=ax), axes=ax).real.reshape(3, -1)
    h += np.einsum("ijx,jx->ix", A - B, phi)
    den = (phi * phi).sum(1)
    mu = (phi * h).sum(1) / np.where(den > 0, den, 1.0)
    if den[1] < 1e-20 * den.sum():
        mu[1] = 0.5 * (mu[0] + mu[2])
    for j in range(3):
        A[j, j] -= mu[j]
    return A


def exact(case, seed):
    c, do = case, case["do"]
    if do == "gram":
        s = prepare(c, seed)
        A, B = (torch.view_as_real(s[x].to(torch.complex128)).permute(0, 2, 1).reshape(-1, c["n"]) for x in "AB")
        return A @ B.T
    if do == "apply":
        s, n = prepare(c, seed), _grid(c)
        phi = _spinor(c, seed).reshape(3, -1)
        A, B = _blocks(c, phi)
        A, B = (torch.from_numpy(m).cuda() for m in (_minus_mu(c, phi, A, B), B))
        k2 = torch.from_numpy(_symbol(c)).cuda()
        ax = tuple(range(1, 1 + len(n)))
        y = torch.empty(s["x"].shape, dtype=torch.complex128, device="cuda")
        for v in range(c["nvec"]):
            x = s["x"][v].to(torch.complex128)
            kin = torch.fft.ifftn(torch.fft.fftn(x.reshape([6] + n), dim=ax) * k2, dim=ax).reshape(6, -1)
            for i in range(3):
                Ax, Bx = ((m[i, :, None] * x.reshape(2, 3, -1).transpose(0, 1)).sum(0) for m in (A, B))
                if c["form"] == "uv":
                    y[v, i], y[v, 3 + i] = kin[i] + Ax[0] + Bx[1], -(kin[3 + i] + Bx[0] + Ax[1])
                else:
                    y[v, i], y[v, 3 + i] = kin[i] + Ax[0] + Bx[0], kin[3 + i] + Ax[1] - Bx[1]
        return y
    if do == "density":
        s = prepare(c, seed)
        phi = torch.from_numpy(_spinor(c, seed).reshape(3, -1)).cuda()
        out = torch.empty((c["nmode"], c["nt"], 3, phi.shape[1]), dtype=torch.float64, device="cuda")
        for l in range(c["nmode"]):
            u, v = s["UV"][l].to(torch.complex128).reshape(2, 3, -1)
            for t in range(c["nt"]):
                th = float(s["omega"][l] * s["times"][t])
                w = complex(math.cos(th), math.sin(th))
                out[l, t] = (phi + 0.1 * (u * w.conjugate() + v.conj() * w)).abs() ** 2
        return out
    if do == "solve" and not c["ny"]:
        phi, n = _ground(_problem(c))[1].reshape(3, -1), c["nx"]
        A, B = _blocks(c, phi)
        A = _minus_mu(c, phi, A, B)
        F = np.fft.fft(np.eye(n), axis=0)
        T = np.fft.ifft(_symbol(c)[:, None] * F, axis=0).real
        Hp, Hm = (np.block([[np.diag(A[i, j] + s * B[i, j]) + (T if i == j else 0.0) for j in range(3)] for i in range(3)])
                  for s in (1, -1))
        w, Q = np.linalg.eigh(0.5 * (Hp + Hp.T))
        R = Q * np.sqrt(np.maximum(w, 0.0))          # H_+ = R R^T: the eigenvalues of R^T H_- R are omega^2
        w2 = np.linalg.eigvalsh(R.T @ (0.5 * (Hm + Hm.T)) @ R)
        return {"omega": np.sqrt(w2[w2 > 1e-8])[: c["k"]], "nconv": None}
    return None
