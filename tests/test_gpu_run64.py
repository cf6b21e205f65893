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

from paper_0912_4457_gb300.nksign import (  # noqa: E402
    NK_ASYNC, NK_DOUBLE_PASS, NK_EBREAKDOWN, NK_EINVAL, NK_ETIMEOUT, NK_FP64, NK_MIXED, NK_NO_GRAPH, NK_OK, NK_PROFILE,
    Context, NkError,
)

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


def test_solves_in_flight_share_the_chip():
    """Eight contexts' solves on eight streams take less than half the time of the eight one after
    the other: a solve's launch of all its steps leaves room for others on its SMs (its CTAs alone
    fill at most a third of them, so that at least two are resident together)."""
    import time
    dims, k, n = (6, 6, 6, 6), 256, 8
    U = inputs.su3_links(dims, 41)[0]
    ctxs, b, y, streams = [], [], [], []
    for i in range(n):
        c = Context(dims)
        c.load_links(U)
        c.set_mu_mw(0.1, M_W)
        ctxs.append(c)
        b.append(torch.from_numpy(inputs.gaussian_sources(dims, 73 + i)).cuda())
        y.append(torch.zeros_like(b[-1]))
        streams.append(torch.cuda.Stream())
    torch.cuda.synchronize()

    def together():
        for c, x, o, s in zip(ctxs, b, y, streams):
            c.sign_apply_dev(x, o, 1, k, 32, flags=NK_FP64 | NK_ASYNC, stream=s)
        for c in ctxs:
            c.wait()

    def in_turn():
        for c, x, o, s in zip(ctxs, b, y, streams):
            c.sign_apply_dev(x, o, 1, k, 32, flags=NK_FP64 | NK_ASYNC, stream=s)
            c.wait()

    def best(f):
        f()
        ts = []
        for _ in range(5):
            t = time.perf_counter()
            f()
            ts.append(time.perf_counter() - t)
        return min(ts)

    assert best(together) < 0.5 * best(in_turn)
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("dims,n,k", [((2, 2, 2, 2), 1, 12), ((3, 5, 3, 7), 2, 30), ((4, 4, 4, 4), 12, 64),
                                      ((6, 6, 6, 6), 1, 64), ((8, 8, 8, 8), 2, 32)])
def test_solve_beside_others_gives_the_same_bits(mu, dims, n, k):
    """NK_ASYNC: a launch per half step instead of one for all; the same result, also of a
    double pass and without a graph."""
    ctx, _ = make_ctx(dims, mu)
    b = torch.from_numpy(inputs.gaussian_sources(dims, 72, n_rhs=n)).cuda()
    for flags in (NK_FP64, NK_FP64 | NK_NO_GRAPH, NK_FP64 | NK_DOUBLE_PASS):
        ref, got = torch.zeros_like(b), torch.zeros_like(b)
        ctx.sign_apply_dev(b, ref, n, k, 8, flags=flags)
        ctx.sign_apply_dev(b, got, n, k, 8, flags=flags | NK_ASYNC)
        ctx.wait()
        assert torch.equal(ref, got)
    ctx.close()


@pytest.mark.parametrize("mu", [0.0, 0.3])
def test_profile_times_the_arithmetic_of_the_solve(mu):
    """NK_PROFILE: the bits of the solve without it, fixed and adaptive k (a recurrence continued
    in chunks), and one launch per half step in the classes of the halves."""
    dims, n, k = (4, 4, 4, 4), 2, 128
    ctx, _ = make_ctx(dims, mu)
    b = inputs.gaussian_sources(dims, 74, n_rhs=n)
    for tol in (0.0, 1e-30):
        y, _, _ = ctx.sign_apply(b, k, 32, tol=tol, check=False)
        yp, st, _ = ctx.sign_apply(b, k, 32, tol=tol, flags=NK_FP64 | NK_PROFILE, check=False)
        np.testing.assert_array_equal(y, yp)
        assert st["n_class"]["dslash64"] == k and st["n_class"]["step2"] == k - 1
        assert st["t_class_ms"]["dslash64"] > 0.0 and st["t_class_ms"]["step2"] > 0.0
    ctx.close()


def test_a_wait_that_runs_out_is_a_timeout_in_every_call():
    """With a limit of 0 the first CTA at a grid barrier gives up: every call that runs the steps
    in one launch reports NK_ETIMEOUT (not success, not a breakdown), and the context goes on
    with the next limit."""
    from paper_0912_4457_gb300 import nksign
    dims, n, k = (6, 6, 6, 6), 2, 64
    ctx, _ = make_ctx(dims, 0.2)
    b = inputs.gaussian_sources(dims, 75, n_rhs=n)
    bd = torch.from_numpy(b).cuda()
    ref, _, _ = ctx.sign_apply(b, k, 16)
    ctx.set_wait_limit(0.0)
    for flags in (NK_FP64, NK_FP64 | NK_NO_GRAPH):
        y, st, rc = ctx.sign_apply(b, k, 16, flags=flags, check=False)
        assert rc == NK_ETIMEOUT and list(st["status"][:n]) == [NK_ETIMEOUT] * n
        assert not y.any()
        assert "wait" in nksign.load_library().nk_last_error(ctx.h).decode()
    y, st, rc = ctx.sign_apply(b, k, 16, tol=1e-8, check=False)
    assert rc == NK_ETIMEOUT and list(st["status"][:n]) == [NK_ETIMEOUT] * n
    with pytest.raises(NkError) as e:
        ctx.outer_lanczos_dev(bd, n, k)
    assert e.value.code == NK_ETIMEOUT
    assert ctx.eigs_smallest(b[0], k, 4, check=False)[-1] == NK_ETIMEOUT
    for bad in (-1.0, 11.0, float("nan")):
        with pytest.raises(NkError) as e:
            ctx.set_wait_limit(bad)
        assert e.value.code == NK_EINVAL
    ctx.set_wait_limit(1.0)
    np.testing.assert_array_equal(ctx.sign_apply(b, k, 16)[0], ref)
    ctx.close()


def test_setting_the_shape_a_context_reports_changes_nothing():
    """nk_set_launch of what nk_get_launch gives keeps the one launch of all steps (same bits, same
    number of launches); another shape takes the step kernels."""
    dims, n, k = (4, 4, 4, 4), 2, 64
    ctx, _ = make_ctx(dims, 0.2)
    b = inputs.gaussian_sources(dims, 76, n_rhs=n)
    y0, st0, _ = ctx.sign_apply(b, k, 16)
    shape = list(ctx.get_launch(n, NK_FP64))
    ctx.set_launch(n, NK_FP64, *shape)
    y1, st1, _ = ctx.sign_apply(b, k, 16)
    assert st1["launches"] == st0["launches"]
    np.testing.assert_array_equal(y0, y1)
    shape[2] += 1
    ctx.set_launch(n, NK_FP64, *shape)
    _, st2, _ = ctx.sign_apply(b, k, 16)
    assert st2["launches"] > st0["launches"] + k
    ctx.close()


def test_autotune_times_the_launch_of_all_steps(tmp_path):
    """Tuning a small FP64 batch keeps the one launch of all steps where that is faster (here by a
    third), in the context that tuned and in one that reads the cache file."""
    dims, n, k = (4, 4, 4, 4), 1, 64
    path = str(tmp_path / "tune.txt")
    b = inputs.gaussian_sources(dims, 77, n_rhs=n)
    ctx, _ = make_ctx(dims, 0.0)
    unset = ctx.get_launch(n, NK_FP64)
    _, st0, _ = ctx.sign_apply(b, k, 16)
    shape, ms = ctx.autotune(n, NK_FP64, path)
    assert shape == unset == ctx.get_launch(n, NK_FP64) and 0.0 < ms < 10.0
    other, _ = make_ctx(dims, 0.0)
    assert other.autotune(n, NK_FP64, path)[0] == unset
    for c in (ctx, other):
        assert c.sign_apply(b, k, 16)[1]["launches"] == st0["launches"]
        c.close()


@pytest.mark.parametrize("dims,n,mu", [((6, 6, 6, 6), 12, 0.3),     # several rounds of both halves, 12 CTAs a source
                                       ((8, 8, 8, 8), 8, 0.0), ((8, 8, 8, 8), 4, 0.3),   # 32768 sites x vectors: one launch
                                       ((8, 8, 8, 8), 9, 0.0), ((8, 8, 8, 8), 5, 0.3)])  # beyond: the step kernels
def test_loops_and_both_sides_of_the_dispatch(dims, n, mu):
    """The first 12 steps against the oracle (1e-11, as in test_gpu_parity), first and last source."""
    k = 12
    ctx, U = make_ctx(dims, mu)
    b = inputs.gaussian_sources(dims, 78, n_rhs=n)
    _, st, _ = ctx.sign_apply(b, k, 8, p=1.0)
    assert (st["launches"] < 2 * k) == (b.shape[1] // 12 * n * (2 if mu else 1) <= 32768)
    al, be, ga, _ = ctx.outer_lanczos_dev(torch.from_numpy(b).cuda(), n, k)
    A, Ad, herm = nested.operator(U, dims, mu, M_W)
    for i in (0, n - 1):
        ref = nested.outer_basis(A, Ad, b[i], k, herm)
        assert rel(al[i], ref.alpha) < 1e-11
        assert rel(be[i, : k - 1], ref.beta[: k - 1]) < 1e-11
        assert rel(ga[i, : k - 1], ref.gamma[: k - 1]) < 1e-11
    ctx.close()


@pytest.mark.parametrize("mu", [0.0, 0.2])
@pytest.mark.parametrize("shape,mixed", [(None, False), ((64, 0, 1), False), ((256, 1, 3), False), (None, True)])
def test_second_pass_regenerates_the_same_bits(mu, shape, mixed):
    """A double-pass solve adds c'_j q_j column by column as the lift of the stored basis does, so with
    a bit-identical second pass the results are equal."""
    dims, n, k = (5, 4, 3, 6), 3, 256
    ctx, _ = make_ctx(dims, mu)
    flags = NK_MIXED if mixed else NK_FP64
    if shape:
        s = list(ctx.get_launch(n, flags))
        s[0], s[1], s[5] = shape
        s[2] += 1
        ctx.set_launch(n, flags, *s)
    b = inputs.gaussian_sources(dims, 79, n_rhs=n)
    y1, _, _ = ctx.sign_apply(b, k, 64, p=1.0, flags=flags)
    y2, _, _ = ctx.sign_apply(b, k, 64, p=1.0, flags=flags | NK_DOUBLE_PASS)
    np.testing.assert_array_equal(y1, y2)
    ctx.close()
