"""The FP64 stencil (16 threads per site): the stencil alone and fused with the
first half of an outer step, on lattices whose volume is no multiple of a
CTA's sites, for every launch shape, and with overlapping input and output.

Tolerances: one application sums about 100 products per component (1e-13);
the first 12 steps of a recurrence agree to 1e-11, as in test_gpu_parity.
"""
import numpy as np
import pytest

import inputs
from oracle import dirac, nested

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300.nksign import NK_DOUBLE_PASS, NK_FP64, Context  # noqa: E402

M_W = -2.0


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def make_ctx(dims, mu, antiperiodic=True):
    U = inputs.su3_links(dims, 41)[0]
    ctx = Context(dims, antiperiodic)
    ctx.load_links(U)
    ctx.set_mu_mw(mu, M_W)
    return ctx, U


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((3, 3, 3, 3), 5), ((2, 3, 5, 7), 24), ((5, 2, 3, 3), 2)])
@pytest.mark.parametrize("antiperiodic", [True, False])
def test_alone_odd_volumes(dims, n, antiperiodic):
    ctx, U = make_ctx(dims, 0.3, antiperiodic)
    x = inputs.gaussian_sources(dims, 42, n_rhs=n)
    xd = torch.from_numpy(x).cuda()
    for dagger in (False, True):
        out = torch.zeros_like(xd)
        ctx.dslash_dev(xd, out, n, dagger=dagger, precision=64)
        got = out.cpu().numpy()
        f = dirac.apply_A_dagger if dagger else dirac.apply_A
        for i in range(n):
            assert rel(got[i], f(x[i], U, dims, 0.3, M_W, antiperiodic_t=antiperiodic)) < 1e-13
    ctx.close()


def test_alone_in_place_and_shifted():
    """out may be in, or overlap it: the result is that of separate arrays."""
    dims, n = (3, 4, 3, 5), 3
    ctx, U = make_ctx(dims, 0.2)
    x = torch.from_numpy(inputs.gaussian_sources(dims, 43, n_rhs=n + 1)).cuda()
    ref = torch.zeros_like(x)
    ctx.dslash_dev(x, ref, n, precision=64)
    for shift in (0, 1):
        buf = x.clone()
        ctx.dslash_dev(buf[:n], buf[shift:shift + n], n, precision=64)
        assert torch.equal(buf[shift:shift + n], ref[:n])
    ctx.close()


@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("threads,order,split", [(64, 0, 1), (128, 1, 1), (256, 0, 1), (64, 1, 3), (128, 0, 3), (256, 1, 3)])
def test_fused_step_shapes(mu, threads, order, split):
    dims, n, k = (3, 5, 3, 7), 2, 12
    ctx, U = make_ctx(dims, mu)
    b = inputs.gaussian_sources(dims, 44, n_rhs=n)
    ctx.set_launch(n, NK_FP64, threads, order, 3, 128, 0, split, 1)
    al, be, ga, _ = ctx.outer_lanczos_dev(torch.from_numpy(b).cuda(), n, k)
    A, Ad, herm = nested.operator(U, dims, mu, M_W)
    for i in range(n):
        ref = nested.outer_basis(A, Ad, b[i], k, herm)
        assert rel(al[i], ref.alpha) < 1e-11
        assert rel(be[i, :k - 1], ref.beta[:k - 1]) < 1e-11
        assert rel(ga[i, :k - 1], ref.gamma[:k - 1]) < 1e-11
    # the second pass of a double-pass solve regenerates the same basis
    y1, _, _ = ctx.sign_apply(b, k, 8, p=1.0)
    y2, _, _ = ctx.sign_apply(b, k, 8, p=1.0, flags=NK_FP64 | NK_DOUBLE_PASS)
    assert rel(y2, y1) < 1e-13
    ctx.close()


def test_operators_back_to_back():
    """Consecutive calls may overlap on the device (dependent launches): a
    chain of applications, each reading the last one's result, equals the same
    chain with a synchronisation after every call, in every precision."""
    dims, n = (5, 4, 3, 6), 3
    ctx, _ = make_ctx(dims, 0.2)
    x = torch.from_numpy(inputs.gaussian_sources(dims, 45, n_rhs=n)).cuda()
    V = int(np.prod(dims))
    f = torch.randn(2 * n, 6, V, 4, device="cuda")

    def chain(sync):
        out = []
        for prec in (64, 48, 32):
            a, b = x.clone(), torch.zeros_like(x)
            for i in range(6):
                ctx.dslash_dev(a, b, n, dagger=bool(i & 1), precision=prec)
                if sync:
                    torch.cuda.synchronize()
                a, b = b, a
            out.append(a.clone())
        p, q = f.clone(), torch.zeros_like(f)
        for i in range(6):
            ctx.stencil32_dev(p, q, n)
            if sync:
                torch.cuda.synchronize()
            p, q = q, p
        out.append(p.clone())
        torch.cuda.synchronize()
        return out
    for u, v in zip(chain(True), chain(False)):
        assert torch.equal(u, v)
    ctx.close()


@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((3, 5, 3, 7), 1), ((3, 3, 4, 5), 5), ((4, 4, 4, 4), 12)])
def test_run_of_steps_matches_step_kernels(mu, dims, n):
    """The cooperative launch of all steps (default shape, small batch) against the oracle and the
    step kernels (a launch shape set), from fewer units of work than CTAs to several per CTA; and
    the adaptive solve, which continues a recurrence in chunks, against the same solve at fixed k."""
    k = 12
    ctx, U = make_ctx(dims, mu)
    b = inputs.gaussian_sources(dims, 46, n_rhs=n)
    bd = torch.from_numpy(b).cuda()
    run = ctx.outer_lanczos_dev(bd, n, k)
    again = ctx.outer_lanczos_dev(bd, n, k)
    for u, v in zip(run, again):
        np.testing.assert_array_equal(u[..., : k - 1], v[..., : k - 1])   # bitwise reproducible
    y2, _, _ = ctx.sign_apply(b, k, 8, p=1.0, flags=NK_FP64 | NK_DOUBLE_PASS)
    y1, _, _ = ctx.sign_apply(b, k, 8, p=1.0)
    assert rel(y2, y1) < 1e-13
    # an adaptive solve that never meets its tolerance continues the recurrence in chunks of 64
    # steps: the arithmetic of a fixed k, step for step
    ya, sta, _ = ctx.sign_apply(b[:1], 128, 32, tol=1e-30, check=False)
    yf, _, _ = ctx.sign_apply(b[:1], 128, 32)
    assert sta["checks"] == 2 and rel(ya, yf) < 1e-12
    ctx.set_launch(n, NK_FP64, 128, 0, 3)
    steps = ctx.outer_lanczos_dev(bd, n, k)
    A, Ad, herm = nested.operator(U, dims, mu, M_W)
    for i in range(n):
        ref = nested.outer_basis(A, Ad, b[i], k, herm)
        for got in (run, steps):
            assert rel(got[0][i], ref.alpha) < 1e-11
            assert rel(got[1][i, : k - 1], ref.beta[: k - 1]) < 1e-11
            assert rel(got[2][i, : k - 1], ref.gamma[: k - 1]) < 1e-11
    ctx.close()


def test_runs_of_two_contexts_in_flight():
    """Two contexts' cooperative launches on two streams: each equals its solve alone."""
    dims, k = (6, 6, 6, 6), 64
    from paper_0912_4457_gb300.nksign import NK_ASYNC
    pair = [make_ctx(dims, 0.2)[0] for _ in range(2)]
    b = [torch.from_numpy(inputs.gaussian_sources(dims, 47 + i)).cuda() for i in range(2)]
    y = [torch.zeros_like(x) for x in b]
    alone = []
    for c, x, o in zip(pair, b, y):
        c.sign_apply_dev(x, o, 1, k, 16)
        alone.append(o.clone())
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(5):
        for c, x, o, s in zip(pair, b, y, streams):
            o.zero_()
            torch.cuda.synchronize()
        for c, x, o, s in zip(pair, b, y, streams):
            c.sign_apply_dev(x, o, 1, k, 16, flags=NK_FP64 | NK_ASYNC, stream=s)
        for c in pair:
            c.wait()
        for o, ref in zip(y, alone):
            assert torch.equal(o, ref)
    for c in pair:
        c.close()
