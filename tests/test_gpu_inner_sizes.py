"""The inner part (inner Lanczos on a cluster, Roberts-Higham iteration) at the
sizes where its layout changes: k around a cluster's lanes (one CTA, 2, 4 and 8
CTAs, two and three rows per lane) and l around the cluster sizes and the
column blocks of the inversion, against the nested oracle.

Ritz matrices: two bands of eigenvalues (diagonal about 0, off-diagonals
alternating 1.44 and 1.26 with 2% noise), complex in the two-sided case.  The tolerance
is that of test_gpu_parity's chunking test: 1e-11, or ten times what rounding-level
changes of H_k move the oracle's own result.
"""
import numpy as np
import pytest

from oracle import nested

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300.nksign import Context  # noqa: E402


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def ritz(n, k, herm, seed):
    rng = np.random.default_rng(seed)
    base = np.where(np.arange(k) % 2 == 0, 1.44, 1.26)
    be = base * (1 + 0.02 * rng.standard_normal((n, k))) + 0j
    al = 0.03 * rng.standard_normal((n, k)) + 0j
    if not herm:
        al = al + 0.03j * rng.standard_normal((n, k))
        be = be * np.exp(0.02j * rng.standard_normal((n, k)))
    ga = be.conj() ** 2 / be
    return al, be, ga


def check(n, k, ell, herm, p, seed=0, rhi_slack=1):
    al, be, ga = ritz(n, k, herm, seed)
    r = (lambda x: x.real) if herm else (lambda x: x)   # the oracle's Hermitian path is real
    ctx = Context((2, 2, 2, 2))
    c, st, _ = ctx.inner_sign(al, be, ga, ell, p=p, hermitian=herm)
    ctx.close()
    for i in range(n):
        h = [r(al[i]), r(be[i, : k - 1]), r(ga[i, : k - 1])]
        pi, zmn, zmx = nested.estimate_p(*h) if p == 0.0 else (p, None, None)
        if p == 0.0:
            assert st["p"][i] == pytest.approx(pi, rel=1e-11)
            assert st["z_min"][i] == pytest.approx(zmn, rel=1e-11)
            assert st["z_max"][i] == pytest.approx(zmx, rel=1e-11)
        ref, info = nested.inner_sign(*h, ell, pi, herm)
        rng = np.random.default_rng(7)
        sens = max(rel(nested.inner_sign(*[x * (1 + 1e-15 * rng.standard_normal(x.shape)) for x in h], ell, pi, herm)[0], ref)
                   for _ in range(2))
        assert rel(c[i], ref) < max(1e-11, 10 * sens)
        assert abs(st["rhi_iters"][i] - info["rhi_iters"]) <= rhi_slack


@pytest.mark.parametrize("herm", [True, False])
@pytest.mark.parametrize("k", [4, 6, 62, 64, 66, 126, 128, 130, 256, 258, 510, 512, 514, 1022, 1024, 1026, 1536])
def test_outer_sizes(k, herm):
    check(2, k, min(k, 24), herm, 0.0 if k >= 64 else 0.9)


@pytest.mark.parametrize("herm", [True, False])
@pytest.mark.parametrize("ell", [2, 6, 14, 16, 18, 30, 34, 62, 64, 66, 98, 128, 160])
def test_inner_sizes(ell, herm):
    check(3, 192, ell, herm, 1.3, seed=ell)


@pytest.mark.parametrize("herm", [True, False])
def test_largest_inner_size(herm):
    check(2, 300, 256, herm, 1.3, seed=9)


@pytest.mark.parametrize("herm", [True, False])
@pytest.mark.parametrize("e", [-900, -200, 300, 900])
def test_power_of_two_scale(e, herm):
    """c depends on p H_k alone: H_k scaled by 2^e with p scaled by 2^-e gives the same bits."""
    al, be, ga = ritz(2, 96, herm, 11)
    ctx = Context((2, 2, 2, 2))
    ref, _, _ = ctx.inner_sign(al, be, ga, 24, p=1.25, hermitian=herm)
    s = 2.0 ** e
    got, _, _ = ctx.inner_sign(al * s, be * s, ga * s, 24, p=1.25 / s, hermitian=herm)
    ctx.close()
    np.testing.assert_array_equal(got, ref)
