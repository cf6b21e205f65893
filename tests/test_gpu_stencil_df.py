"""The two-float stencil with one and with two threads per site and vector: both
sides of the rule that chooses, volumes that are no multiple of a CTA's sites,
half-filled last warps, both boundary conditions, alone and scaled inside a step.

Tolerances: 2e-13 for one application (about 48-bit arithmetic) and 1e-11 for
the first steps of a recurrence, as in test_gpu_parity.
"""
import numpy as np
import pytest

import inputs
from oracle import dirac, nested

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300.nksign import NK_MIXED, Context  # noqa: E402

M_W = -2.0


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def make_ctx(dims, mu, antiperiodic=True):
    U = inputs.su3_links(dims, 51)[0]
    ctx = Context(dims, antiperiodic)
    ctx.load_links(U)
    ctx.set_mu_mw(mu, M_W)
    return ctx, U


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((3, 3, 3, 3), 2), ((2, 3, 5, 7), 6), ((3, 5, 3, 2), 7),
                                    ((3, 3, 3, 5), 8), ((3, 3, 3, 5), 9), ((2, 3, 3, 3), 24)])
@pytest.mark.parametrize("antiperiodic", [True, False])
def test_alone(dims, n, antiperiodic):
    ctx, U = make_ctx(dims, 0.3, antiperiodic)
    x = inputs.gaussian_sources(dims, 52, n_rhs=n)
    xd = torch.from_numpy(x).cuda()
    for dagger in (False, True):
        out = torch.zeros_like(xd)
        ctx.dslash_dev(xd, out, n, dagger=dagger, precision=48)
        got = out.cpu().numpy()
        f = dirac.apply_A_dagger if dagger else dirac.apply_A
        for i in range(n):
            assert rel(got[i], f(x[i], U, dims, 0.3, M_W, antiperiodic_t=antiperiodic)) < 2e-13
    ctx.close()


@pytest.mark.parametrize("dims", [(16, 16, 16, 3), (17, 16, 16, 3)])
@pytest.mark.parametrize("n", [6, 7, 8, 9, 12, 13])
def test_rule_by_sites(dims, n):
    """On both sides of 12288 sites, against the FP64 stencil."""
    ctx, _ = make_ctx(dims, 0.2)
    x = torch.from_numpy(inputs.gaussian_sources(dims, 53, n_rhs=n)).cuda()
    got, ref = torch.zeros_like(x), torch.zeros_like(x)
    ctx.dslash_dev(x, got, n, precision=48)
    ctx.dslash_dev(x, ref, n, precision=64)
    for i in range(n):
        assert rel(got[i].cpu().numpy(), ref[i].cpu().numpy()) < 2e-13
    ctx.close()


@pytest.mark.parametrize("mu,n", [(0.0, 1), (0.0, 8), (0.0, 9), (0.3, 1), (0.3, 3), (0.3, 5)])
def test_inside_a_step(mu, n):
    dims, k = (3, 4, 3, 5), 10
    ctx, U = make_ctx(dims, mu)
    b = inputs.gaussian_sources(dims, 54, n_rhs=n)
    ctx.set_precision(k)
    got = ctx.outer_lanczos_dev(torch.from_numpy(b).cuda(), n, k, flags=NK_MIXED)
    A, Ad, herm = nested.operator(U, dims, mu, M_W)
    for i in range(n):
        ref = nested.outer_basis(A, Ad, b[i], k, herm)
        assert rel(got[0][i], ref.alpha) < 1e-11
        assert rel(got[1][i, : k - 1], ref.beta[: k - 1]) < 1e-11
    ctx.close()
