"""Chains of operator calls whose grids are several waves of the chip: while a call's
last CTAs still write, CTAs of the next call (a dependent launch) are already
placed.  Every link of the chain reads what the one before wrote, so the chain
must equal, bit for bit, the same chain with a synchronisation after every call.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300.nksign import Context  # noqa: E402

DIMS, N = (12, 12, 12, 12), 12   # 2592 CTAs of 8 sites (31104 of the FP64 stencil)


@pytest.fixture(scope="module")
def ctx():
    c = Context(DIMS)
    c.load_links(inputs.su3_links(DIMS, 61)[0])
    c.set_mu_mw(0.2, -2.0)
    yield c
    c.close()


def both(step, a, b, links=8):
    """The chain a -> b -> a ..., synchronised after every call and not."""
    got = []
    for sync in (True, False):
        p, q = a.clone(), b.clone()
        torch.cuda.synchronize()
        for i in range(links):
            step(p, q, i)
            if sync:
                torch.cuda.synchronize()
            p, q = q, p
        torch.cuda.synchronize()
        got.append(p)
    return got


@pytest.mark.parametrize("n", [N, 5])
@pytest.mark.parametrize("precision", [64, 48, 32])
def test_dslash_chain(ctx, precision, n):
    x = torch.from_numpy(inputs.gaussian_sources(DIMS, 62, n_rhs=n)).cuda()
    for _ in range(3):
        u, v = both(lambda p, q, i: ctx.dslash_dev(p, q, n, dagger=bool(i & 1), precision=precision), x,
                    torch.zeros_like(x))
        assert torch.equal(u, v)


@pytest.mark.parametrize("n", [N, 5])
def test_stencil32_chain(ctx, n):
    V = int(np.prod(DIMS))
    f = torch.randn(2 * n, 6, V, 4, device="cuda", generator=torch.Generator("cuda").manual_seed(63))
    for _ in range(3):
        u, v = both(lambda p, q, i: ctx.stencil32_dev(p, q, n), f, torch.zeros_like(f))
        assert torch.equal(u, v)
