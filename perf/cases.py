"""Timed cases of the library: what a user's program calls, over the sizes it calls it with.

Kinds of case (the key "kind" and the public call it makes):

  apply      Context.dslash_dev     A or A^dagger on device vectors, 64 bits or two-float (48)
  stencil32  Context.stencil32_dev  the FP32 stencil in its native layout, A and A^dagger together
  basis      Context.outer_lanczos_dev  the (two-sided) Lanczos coefficients H_k of device sources
  inner      Context.inner_sign     c = V_l sgn(H_l) e_1 of given Ritz matrices (host arrays)
  sign       Context.sign_apply_dev y = sgn(A) b on device tensors
  overlap    Context.overlap_apply  D_ov b on host arrays

Lattices, sources and parameters are synthetic: links U = exp(i EPS X) with X a random traceless
Hermitian matrix (mean plaquette about 0.59), m_w = -2, Gaussian or point sources.  Sizes are those
of this repository's benchmark and tests (4^4 to 10^4 and 16^3 x 32) and generic ones between them.
Whole solves use subspace sizes at which the result has converged, so that it does not depend on
the rounding of the (not reorthogonalised) recurrences.
"""
import math

import numpy as np
import torch

import paper_0912_4457_gb300 as nk
from paper_0912_4457_gb300 import nksign

M_W = -2.0
KAPPA = 1.0 / (8.0 + 2.0 * M_W)
EPS = 0.4394        # mean plaquette 0.59 on large lattices
DEV = "cuda"


# ---- the cases ------------------------------------------------------------------

def listed():
    return [
        # the smallest call: A on one vector of the smallest lattice (a residual check, a power
        # iteration of a user's own): latency and launches
        dict(name="apply64_4x4x4x4_1", kind="apply", dims="4x4x4x4", mu=0.3, n=1, dagger=False, precision=64),
        # A^dagger in 64 bits on the 12 columns of a propagator, largest lattice
        dict(name="apply64_16x16x16x32_12", kind="apply", dims="16x16x16x32", mu=0.2, n=12, dagger=True, precision=64),
        # the two-float operator on an odd lattice and a ragged number of vectors
        dict(name="apply48_9x9x9x11_7", kind="apply", dims="9x9x9x11", mu=0.2, n=7, dagger=False, precision=48),
        # the FP32 stencil of the late outer steps, 12 right-hand sides: largest lattice (HBM)
        # and the benchmark's 10^4 (operands partly in L2)
        dict(name="stencil32_16x16x16x32_12", kind="stencil32", dims="16x16x16x32", mu=0.2, n=12),
        dict(name="stencil32_10x10x10x10_12", kind="stencil32", dims="10x10x10x10", mu=0.2, n=12),
        # the first steps of the two-sided recurrence from one Gaussian source (Ritz values for
        # choosing k and l, a look at the spectrum)
        dict(name="basis64_6x6x6x6_k64", kind="basis", dims="6x6x6x6", mu=0.3, n=1, k=64),
        # the inner half alone on 12 two-sided Ritz matrices at the benchmark's k and l
        dict(name="inner_k1024_l128_12", kind="inner", n=12, k=1024, ell=128, hermitian=False),
        # one Gaussian source, Hermitian, all FP64: the smallest whole solve
        dict(name="sign64_4x4x4x4_k256", kind="sign", dims="4x4x4x4", mu=0.0, n=1, k=256, ell=64, ell2=0,
             mixed=False, j0=-1, double_pass=False, source="gauss"),
        # one Gaussian source, non-Hermitian, all FP64
        dict(name="sign64_6x6x6x6_k512", kind="sign", dims="6x6x6x6", mu=0.1, n=1, k=512, ell=128, ell2=0,
             mixed=False, j0=-1, double_pass=False, source="gauss"),
        # the overlap operator on the 12 point sources, Hermitian, mixed precision, host arrays
        dict(name="overlap_8x8x8x8_k768_12", kind="overlap", dims="8x8x8x8", mu=0.0, n=12, k=768, ell=160, mixed=True),
        # the plain method: one point source at a time, all FP64, at the benchmark's lattice and sizes
        dict(name="sign64_10x10x10x10_k1024", kind="sign", dims="10x10x10x10", mu=0.2, n=1, k=1024, ell=128, ell2=0,
             mixed=False, j0=-1, double_pass=False, source="point"),
        # the benchmark's batch: 12 point sources, mixed precision, a second nested level
        dict(name="sign_10x10x10x10_k1024_12", kind="sign", dims="10x10x10x10", mu=0.2, n=12, k=1024, ell=128, ell2=64,
             mixed=True, j0=512, double_pass=False, source="point"),
    ]


def _even(x):
    return 2 * int(round(x / 2))


def _draw_dims(rng, vmin, vmax):
    """Four extents, odd ones among them, the volume spread over the logarithm of [vmin, vmax]."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    while True:
        ext = [max(2, int(round(target ** 0.25 * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(4)]
        if vmin <= math.prod(ext) <= vmax:
            return ext


def _name(ext):
    return "x".join(str(e) for e in ext)


def draw(rng):
    kind = rng.choice(["apply", "stencil32", "basis", "inner", "sign", "sign", "overlap"])
    if kind == "apply":
        ext = _draw_dims(rng, 256, 131072)
        return dict(kind=kind, dims=_name(ext), mu=round(rng.uniform(0.0, 0.3), 3), n=rng.randint(1, 12),
                    dagger=rng.random() < 0.5, precision=rng.choice([64, 64, 48]))
    if kind == "stencil32":
        ext = _draw_dims(rng, 256, 131072)
        return dict(kind=kind, dims=_name(ext), mu=round(rng.uniform(0.0, 0.3), 3), n=rng.randint(1, 12))
    if kind == "basis":
        ext = _draw_dims(rng, 256, 10000)
        return dict(kind=kind, dims=_name(ext), mu=rng.choice([0.0, round(rng.uniform(0.05, 0.3), 3)]),
                    n=rng.randint(1, 12), k=2 * rng.randint(8, 40))
    if kind == "inner":
        k = _even(math.exp(rng.uniform(math.log(128), math.log(1024))))
        return dict(kind=kind, n=rng.randint(1, 12), k=k, ell=max(48, min(128, _even(k * rng.uniform(0.125, 0.3)))),
                    hermitian=rng.random() < 0.5)
    while True:
        ext = _draw_dims(rng, 512, 8192)
        v = math.prod(ext)
        n = rng.randint(1, 12)
        mu = 0.0 if kind == "overlap" else rng.choice([0.0, round(rng.uniform(0.02, 0.08), 3)])
        mixed = rng.random() < 0.5
        double_pass = kind == "sign" and rng.random() < 0.25
        k = _even((640 if v <= 1024 else 768 if v <= 4096 else 960) * rng.uniform(1.0, 1.2))
        # no dearer than the largest listed case (12 sources of 10^4 sites, two-sided, mixed)
        cost = n * v * k * (1 if mu == 0.0 else 2) * (2 if double_pass else 1) * (1 if mixed else 2.5)
        if cost <= 12 * 10000 * 1024 * 2 * 0.8:
            break
    ell = _even(k * rng.uniform(0.2, 0.25))
    if kind == "overlap":
        return dict(kind=kind, dims=_name(ext), mu=0.0, n=n, k=k, ell=ell, mixed=mixed)
    return dict(kind=kind, dims=_name(ext), mu=mu, n=n, k=k, ell=ell, ell2=rng.choice([0, _even(ell * 0.6)]), mixed=mixed,
                j0=_even(k * (0.4 if mu == 0.0 else 0.75)) if mixed else -1, double_pass=double_pass,
                source=rng.choice(["gauss", "point"]))


# ---- inputs ---------------------------------------------------------------------

def _dims(case):
    return tuple(int(x) for x in case["dims"].split("x"))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randc(g, *shape):
    return torch.complex(torch.randn(*shape, generator=g, dtype=torch.float64, device=DEV),
                         torch.randn(*shape, generator=g, dtype=torch.float64, device=DEV)) / math.sqrt(2.0)


def _links(dims, g):
    """[t][z][y][x][nu][3][3] complex128 links exp(i EPS X)."""
    x, y, z, t = dims
    a = _randc(g, t * z * y * x * 4, 3, 3)
    h = 0.5 * (a + a.mH)
    tr = h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3.0
    h = h - tr[:, None, None] * torch.eye(3, dtype=torch.complex128, device=DEV)
    return torch.linalg.matrix_exp(1j * EPS * h).reshape(t, z, y, x, 4, 3, 3).contiguous()


def _sources(case, dims, g):
    """(n, 12 V) complex128: Gaussian vectors, or spin-colour point sources at one site."""
    n, N = case["n"], 12 * math.prod(dims)
    if case.get("source") == "point" or case["kind"] == "overlap":
        site = int(torch.randint(0, N // 12, (1,), generator=g, device=DEV))
        b = torch.zeros(n, N, dtype=torch.complex128, device=DEV)
        for i in range(n):
            b[i, 12 * site + i] = 1.0
        return b
    return _randc(g, n, N)


def _ritz(case, g):
    """alpha, beta, gamma (n, k): Ritz matrices with the structure the outer recurrence gives here:
    a small diagonal and off-diagonals alternating about 1.44 and 1.28 (a spectrum of two bands
    [-2.8, -0.15] and [0.15, 2.8]); two-sided: complex entries, gamma = (beta^*)^2 / beta."""
    n, k = case["n"], case["k"]
    base = torch.where(torch.arange(k, device=DEV) % 2 == 0, 1.44, 1.26).to(torch.float64)
    beta = base * (1.0 + 0.02 * torch.randn(n, k, generator=g, dtype=torch.float64, device=DEV))
    alpha = 0.03 * torch.randn(n, k, generator=g, dtype=torch.float64, device=DEV)
    if case["hermitian"]:
        alpha, beta = alpha.to(torch.complex128), beta.to(torch.complex128)
        gamma = beta.clone()
    else:
        alpha = torch.complex(alpha, 0.03 * torch.randn(n, k, generator=g, dtype=torch.float64, device=DEV))
        beta = torch.polar(beta, 0.02 * torch.randn(n, k, generator=g, dtype=torch.float64, device=DEV))
        gamma = beta.conj() ** 2 / beta
    beta[:, -1] = 0.0
    gamma[:, -1] = 0.0
    return [t.cpu().numpy() for t in (alpha, beta, gamma)]


def _context(case, dims, U):
    c = nk.Context(dims)
    c.load_links_dev(U)
    c.set_mu_mw(case["mu"], M_W)
    return c


def _flags(case):
    f = nk.NK_MIXED if case["mixed"] else nk.NK_FP64
    if case["n"] > 1:
        f |= nksign.NK_SHARED_P
    if case.get("double_pass"):
        f |= nksign.NK_DOUBLE_PASS
    return f


def prepare(case, seed):
    g = _gen(seed)
    if case["kind"] == "inner":
        c = nk.Context((2, 2, 2, 2))
        return dict(case=case, ctx=c, H=_ritz(case, g))
    dims = _dims(case)
    V, n = math.prod(dims), case["n"]
    U = _links(dims, g)
    c = _context(case, dims, U)
    s = dict(case=case, ctx=c)
    if case["kind"] == "stencil32":
        s["in"] = torch.randn(2 * n, 6, V, 4, generator=g, dtype=torch.float32, device=DEV)
        s["out"] = torch.empty_like(s["in"])
        return s
    s["b"] = _sources(case, dims, g)
    if case["kind"] == "overlap":
        s["b"] = s["b"].cpu().numpy()
        return s
    s["y"] = torch.empty_like(s["b"])
    if case["kind"] == "sign":
        c.set_nesting((case["ell2"],) if case["ell2"] else ())
        c.set_precision(case["j0"])
    return s


def run(s):
    case, c = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "apply":
        c.dslash_dev(s["b"], s["y"], case["n"], dagger=case["dagger"], precision=case["precision"])
        return s["y"]
    if kind == "stencil32":
        c.stencil32_dev(s["in"], s["out"], case["n"])
        return s["out"]
    if kind == "basis":
        al, be, ga, xn = c.outer_lanczos_dev(s["b"], case["n"], case["k"])
        return al, be[:, :-1], ga[:, :-1], xn
    if kind == "inner":
        return c.inner_sign(*s["H"], case["ell"], hermitian=case["hermitian"])[0]
    if kind == "overlap":
        return c.overlap_apply(s["b"], case["k"], case["ell"], flags=_flags(case))[0]
    c.sign_apply_dev(s["b"], s["y"], case["n"], case["k"], case["ell"], flags=_flags(case))
    return s["y"]


# ---- what a pass cannot do without -------------------------------------------------

def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "inner":
        k, ell = case["k"], case["ell"]
        e = 2 if case["hermitian"] else 8           # flops of a multiply-add, real or complex
        # l applications of H' (band product and solve, both sides two-sided: about 12 multiply-adds
        # a row), the l x l inverses of about 7 Roberts-Higham steps, the lift V_l s
        sides = 1 if case["hermitian"] else 2
        flops = n * e * (sides * 12.0 * ell * k + 7.0 * ell ** 3 + ell * k)
        return dict(bytes=16.0 * n * 4 * k, flops=flops)
    V = math.prod(_dims(case))
    N = 12 * V
    if kind == "apply":
        return dict(bytes=16.0 * (36 * V + 2 * n * N), flops=1320.0 * V * n)
    if kind == "stencil32":
        return dict(bytes=8.0 * (36 * V + 2 * 2 * n * N), flops=1320.0 * V * 2 * n)
    k = case["k"]
    sides = 1 if case["mu"] == 0.0 else 2
    # an outer step per source: the stencil on each side, three updates and inner products
    step = V * (1320.0 * sides) + N * (24.0 if sides == 1 else 48.0)
    if kind == "basis":
        return dict(bytes=16.0 * (36 * V + n * N + 3 * n * k), flops=n * k * step)
    # a whole solve also writes the basis once, reads it once for the lift, and lifts
    basis = 0.0 if case.get("double_pass") else 2.0 * 16.0 * n * k * N
    passes = 2 if case.get("double_pass") else 1
    return dict(bytes=16.0 * (36 * V + 2 * n * N) + basis, flops=n * k * (passes * step + 8.0 * N))


# ---- the same in plain torch, 64 bits ---------------------------------------------

# gamma_nu psi in the chiral basis: spin row s of the result is phase[s] psi[perm[s]]
_GAMMA = [((3, 2, 1, 0), (-1j, -1j, 1j, 1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
          ((2, 3, 0, 1), (-1j, 1j, 1j, -1j)), ((2, 3, 0, 1), (1, 1, 1, 1))]


class _Dirac:
    """A = gamma5 D_w(mu) and A^dagger on (n, 12 V) complex128 vectors."""

    def __init__(self, dims, U, mu):
        self.shape = tuple(reversed(dims)) + (4, 3)
        self.mu = mu
        self.U = [U[..., nu, :, :].clone() for nu in range(4)]
        self.U[3][-1] *= -1.0                      # antiperiodic in t
        self.U = [u.unsqueeze(-3) for u in self.U]
        self.Ud = [u.mH.resolve_conj().contiguous() for u in self.U]
        self.phase = [torch.tensor(ph, dtype=torch.complex128, device=DEV)[:, None] for _, ph in _GAMMA]

    def __call__(self, v, dagger=False):
        out = torch.empty_like(v)
        mu = -self.mu if dagger else self.mu
        for i in range(v.shape[0]):
            p = v[i].reshape(self.shape)
            acc = torch.zeros_like(p)
            for nu in range(4):
                ax = 3 - nu
                wp, wm = (math.exp(mu), math.exp(-mu)) if nu == 3 else (1.0, 1.0)
                perm = list(_GAMMA[nu][0])
                h = p + self.phase[nu] * p[..., perm, :]                       # (1 + gamma) psi
                acc += wp * torch.roll((self.U[nu] * h.unsqueeze(-2)).sum(-1), 1, ax)
                q = torch.roll(p, -1, ax)
                h = q - self.phase[nu] * q[..., perm, :]                       # (1 - gamma) psi
                acc += wm * (self.Ud[nu] * h.unsqueeze(-2)).sum(-1)
            r = p - KAPPA * acc
            r[..., 2:, :] *= -1.0                  # gamma5
            out[i] = r.reshape(-1)
        return out


def _sign_exact(A, b, k):
    """sgn(A) b by Arnoldi with full reorthogonalisation and Newton's iteration for sgn(H)."""
    n, N = b.shape
    k = min(k, N)
    V = torch.zeros(n, k, N, dtype=torch.complex128, device=DEV)
    H = torch.zeros(n, k, k, dtype=torch.complex128, device=DEV)
    nrm = torch.linalg.vector_norm(b, dim=1)
    V[:, 0] = b / nrm[:, None]
    for j in range(k):
        w = A(V[:, j].contiguous())
        for i in range(n):
            Vj = V[i, : j + 1]
            for _ in range(2):
                h = torch.mv(Vj, w[i].conj()).conj()
                H[i, : j + 1, j] += h
                w[i] -= torch.mv(Vj.T, h)
        if j + 1 < k:
            s = torch.linalg.vector_norm(w, dim=1)
            H[:, j + 1, j] = s
            V[:, j + 1] = w / s[:, None]
    S = H
    for _ in range(60):
        S1 = 0.5 * (S + torch.linalg.inv(S))
        d = float(torch.linalg.matrix_norm(S1 - S).max() / torch.linalg.matrix_norm(S1).max())
        S = S1
        if d < 1e-13:
            break
    c = S[:, :, 0] * nrm[:, None]
    return torch.bmm(c.unsqueeze(1), V).squeeze(1)


def _lanczos_exact(A, b, k, two_sided):
    """The coefficients of the (two-sided) Lanczos recurrence, one source after the other."""
    n = b.shape[0]
    al = torch.zeros(n, k, dtype=torch.complex128)
    be, ga = torch.zeros(n, k, dtype=torch.complex128), torch.zeros(n, k, dtype=torch.complex128)
    nrm = torch.linalg.vector_norm(b, dim=1)
    for r in range(n):
        v = b[r: r + 1] / nrm[r]
        w = v.clone()
        v0 = w0 = torch.zeros_like(v)
        bj = gj = 0.0
        for j in range(k):
            x = A(v) - gj * v0
            a = complex(torch.sum(w.conj() * x))
            if not two_sided:
                a = a.real
            x = x - a * v
            al[r, j] = a
            if j == k - 1:
                break
            if two_sided:
                l = A(w, True) - np.conj(bj) * w0 - np.conj(a) * w
                d = complex(torch.sum(x.conj() * l))
                bj = complex(np.sqrt(np.complex128(d)))
                gj = np.conj(d) / bj
                v0, w0, v, w = v, w, x / bj, l / np.conj(gj)
            else:
                bj = gj = float(torch.linalg.vector_norm(x))
                v0, v = v, x / bj
                w = v
            be[r, j], ga[r, j] = bj, gj
    return al, be, ga, nrm.cpu()


def _inner_exact(case, H):
    """sgn(H_k) e_1 of the whole Ritz matrices."""
    al, be, ga = [torch.from_numpy(x).to(DEV) for x in H]
    k = case["k"]
    M = torch.diag_embed(al) + torch.diag_embed(be[:, : k - 1], -1) + torch.diag_embed(ga[:, : k - 1], 1)
    for _ in range(60):
        M1 = 0.5 * (M + torch.linalg.inv(M))
        d = float(torch.linalg.matrix_norm(M1 - M).max() / torch.linalg.matrix_norm(M1).max())
        M = M1
        if d < 1e-13:
            break
    return M[:, :, 0].contiguous()


def exact(case, seed):
    g = _gen(seed)
    kind, n = case["kind"], case["n"]
    if kind == "inner":
        if n * case["k"] ** 3 > 1.4e10:
            return None
        return _inner_exact(case, _ritz(case, g))
    dims = _dims(case)
    V = math.prod(dims)
    N = 12 * V
    U = _links(dims, g)
    A = _Dirac(dims, U, case["mu"])
    if kind == "stencil32":
        x = torch.randn(2 * n, 6, V, 4, generator=g, dtype=torch.float32, device=DEV)
        A = _Dirac(dims, U.to(torch.complex64).to(torch.complex128), case["mu"])   # the links the stencil holds

        def to_abi(p):      # [6][V] of (re, im, re, im) -> [V][12]
            return torch.view_as_complex(p.to(torch.float64).reshape(n, 6, V, 2, 2).contiguous()).permute(0, 2, 1, 3).reshape(n, N)

        def to_pair(v):
            return torch.view_as_real(v.reshape(n, V, 6, 2).permute(0, 2, 1, 3).contiguous()).reshape(n, 6, V, 4)
        return torch.cat([to_pair(A(to_abi(x[:n]))), to_pair(A(to_abi(x[n:]), True))])
    b = _sources(case, dims, g)
    if kind == "apply":
        return A(b, case["dagger"])
    if kind == "basis":
        if n * case["k"] > 160:
            return None
        al, be, ga, nrm = _lanczos_exact(A, b, case["k"], case["mu"] != 0.0)
        return al, be[:, :-1], ga[:, :-1], nrm
    if n * float(case["k"]) ** 2 * N > 1.2e10:      # some seconds of FP64 arithmetic, and the basis in memory
        return None
    y = _sign_exact(A, b, case["k"])
    if kind == "overlap":
        gy = y.reshape(n, V, 4, 3).clone()
        gy[:, :, 2:] *= -1.0
        return b + gy.reshape(n, N)
    return y
