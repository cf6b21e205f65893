"""The cooperative launch that runs the FP64 steps of a small batch (k_run64): its
ways out, and the sizes where its dispatch and its loops change.
"""
import numpy as np
import pytest

import inputs
from oracle import nested

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300.nksign import NK_EBREAKDOWN, NK_FP64, NK_OK, Context  # noqa: E402

M_W = -2.0


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def make_ctx(dims, mu):
    U = inputs.su3_links(dims, 41)[0]
    ctx = Context(dims)
    ctx.load_links(U)
    ctx.set_mu_mw(mu, M_W)
    return ctx, U


def test_breakdown_of_one_source_of_a_batch():
    """Source 0 is an eigenvector of the free field (its first residual is zero): every CTA of that
    source leaves at the first step, which is a breakdown and never a timeout, and source 1 of the
    batch goes on (8 steps, against the oracle)."""
    dims, k, ell = (4, 4, 4, 4), 8, 4
    ctx = Context(dims, bc_t_antiperiodic=False)
    U = inputs.unit_links(dims)
    ctx.load_links(U)
    ctx.set_mu_mw(0.0, M_W)
    b = np.zeros((2, 12 * 256), complex)
    b[0, 0::12] = 1.0
    b[1] = inputs.gaussian_sources(dims, 71)[0]
    ref = nested.sign_apply(U, dims, 0.0, M_W, b[1], k, ell, p=1.0, antiperiodic_t=False)[0]
    for _ in range(20):
        y, st, rc = ctx.sign_apply(b, k, ell, p=1.0, flags=NK_FP64, check=False)
        assert rc == NK_EBREAKDOWN
        assert list(st["status"][:2]) == [NK_EBREAKDOWN, NK_OK]
        assert not y[0].any()
        assert rel(y[1], ref) < 1e-10
    ctx.close()
