"""Grids in extreme units.  A grid whose lengths are scaled by a power of two scales every operator
coefficient by a power of two exactly, so that what a call computes differs from the unscaled call's by
that power and nothing else, as long as the arithmetic keeps its range."""
import numpy as np
import pytest

from helpers import mg_params, rel_l2, to_gpu, to_np
from paper_1012_4307_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def helm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_4307_gb300 import helm as H
    H.load()
    return H


def handle(helm, n, k2, power, layers=0.75, **kw):
    """A handle on [-2^power, 2^power]^dim; k2 is that of the unscaled grid."""
    dim, s = len(n), 2.0 ** power
    return helm.helm_create(dim, list(n), torch.from_numpy(np.ascontiguousarray(k2 / s ** 2)).cuda(), lo=[-s] * dim,
                            hi=[s] * dim, r0_lo=[-layers * s] * dim, r0_hi=[layers * s] * dim, mg=mg_params(helm, **kw))


@pytest.mark.parametrize("power", [-90, 90])
def test_fp64_gram_schmidt_keeps_its_range(helm, power):
    """Unpreconditioned FGMRES in FP64: w = A v is about 1e57 or 1e-51 and its second-pass corrections some
    16 digits below, outside the range of FP32 on either side.  The scaled solve is the unscaled one: the
    same arithmetic up to a power of two but for the last place of the moduli (hypot), which a residual
    history of some 60 steps carries at below 1e-10 of the right-hand side; both end at 1e-10."""
    n = 33
    k2 = W.k2_well_growth(2, n, kh_max=0.3)
    f = to_gpu(W.random_box_source(2, n, 5))
    out = []
    for p in (0, power):
        h = handle(helm, (n, n), k2, p, pc="none", prec="c128", gs="fp64")
        x, st = helm.krylov_solve(h, f, tol=1e-10, restart=64, maxit=6000, history=True)
        assert st.status == helm.HELM_OK and st.rel_res <= 1e-10 and st.reorthogonalizations > 0
        out.append((x * 2.0 ** (-2 * p), st))
    (x0, st0), (x1, st1) = out
    m = min(60, st0.iterations, st1.iterations)
    assert np.max(np.abs(np.array(st0.history[:m]) - np.array(st1.history[:m]))) <= 1e-10
    assert abs(st0.iterations - st1.iterations) <= 1
    # both residuals are at most 1e-10 of f: the solutions differ by at most the condition number times
    # twice that (|A| up to 8 / h^2, smallest eigenvalue of size 1)
    assert float(torch.linalg.vector_norm(x1 - x0) / torch.linalg.vector_norm(x0)) <= 2e-10 * 8 / (2 / 32) ** 2


@pytest.mark.parametrize("power", [0, -90, 90])
def test_fp64_gram_schmidt_with_large_second_corrections(helm, power):
    """A right-hand side that is an eigenvector up to 1e-8: the first orthogonalisation cancels eight digits,
    and the second pass's correction, the rounding left behind, is some 1e-8 of what remains, far above the
    bound for the short form.  Against a dense solve."""
    n = 17
    h = handle(helm, (n, n), np.zeros((n, n)), power, layers=2.0, pc="none", prec="c128", gs="fp64")
    s = np.sin(np.pi * np.arange(n) / (n - 1))
    s[-1] = 0.0
    f = np.outer(s, s) + 1e-8 * W.random_field((n, n), 6)
    f /= np.linalg.norm(f)
    x, st = helm.krylov_solve(h, to_gpu(f), tol=1e-11, restart=60, maxit=600, history=True)
    assert st.status == helm.HELM_OK and st.reorthogonalizations > 0
    m = n - 2
    lap = (2 * np.eye(m) - np.eye(m, k=1) - np.eye(m, k=-1)) * ((n - 1) / 2.0) ** 2
    A = np.kron(np.eye(m), lap) + np.kron(lap, np.eye(m))
    ref = np.linalg.solve(A, f[1:-1, 1:-1].ravel())
    # condition number about 100, residual at most 1e-11
    assert rel_l2(to_np(x)[1:-1, 1:-1].ravel() * 2.0 ** (-2 * power), ref) <= 2e-9


@pytest.mark.parametrize("n,power,smoother,nu,tail", [
    ((49, 49), -26, "jacobi", (1, 2), 0), ((49, 49), -26, "rb", (1, 1), 0),       # level tiles
    ((49, 49), -26, "jacobi", (1, 2), -1), ((49, 49), -26, "rb", (1, 1), -1),     # cluster tail
    ((49, 49), -26, "jacobi", (2, 2), -1), ((21, 21, 21), -27, "jacobi", (1, 1), -1),
])
def test_complex64_diagonals_keep_their_range(helm, n, power, smoother, nu, tail):
    """Diagonals of about 1e19, whose squared moduli are just below the largest float (between 2^126 and
    2^128): their reciprocals are formed by a division, not by an approximation that gives 0 there.  The
    scaled cycle is the unscaled one up to complex64 rounding (the reciprocal of a squared modulus is a
    subnormal with 22 bits here): the bound of the other complex64 cycles, 2e-5."""
    dim = len(n)
    k2 = W.k2_well_growth(dim, n[0], kh_max=0.3)
    v = to_gpu(W.random_field(tuple(reversed(n)), 7))
    out = []
    for p in (0, power):
        h = handle(helm, n, k2, p, prec="c64", smoother=smoother, nu=nu, coarsest_n=13 if dim == 2 else 7)
        if tail >= 0:
            helm.helm_set_tuning(h, dict(tail_levels=tail))
        out.append(to_np(helm.mg_precondition(h, v)).astype(np.complex128) * 2.0 ** (-2 * p))
    assert rel_l2(out[1], out[0]) <= 2e-5
