"""Kernels that are chosen by size, precision or smoother, at the edges of their ranges, against the
oracle's cycle: the same bounds as the per-level kernels (1e-12 in complex128: a cycle's roundings
amplified by the coarsest solve; 2e-5 in complex64)."""
import numpy as np
import pytest

from helpers import gpu_handle, oracle_pair, rel_l2, to_gpu, to_np
from paper_1012_4307_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {"c128": 1e-12, "c64": 2e-5}


@pytest.fixture(scope="module")
def helm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_4307_gb300 import helm as H
    H.load()
    return H


def problem(n, coarsest_n):
    """Nodes n per axis (x first); k^2 cut from the square or cubic well field."""
    dim = len(n)
    k2 = W.k2_well_growth(dim, max(n), kh_max=0.5)[tuple(slice(0, m) for m in reversed(n))]
    shape = tuple(reversed(n))
    return W.Problem("paths", dim, list(n), np.ascontiguousarray(k2), np.zeros(shape, complex), coarsest_n=coarsest_n)


def check_cycle(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma, tunings=({},), omega=0.8, pc="csg"):
    P = problem(n, coarsest_n)
    h = gpu_handle(helm, P, pc=pc, prec=prec, smoother=smoother, nu=nu, gamma=gamma, omega=omega)
    A, M = oracle_pair(oracle, P, pc=pc)
    v = W.random_field(tuple(reversed(n)), 51)
    ref = oracle.MG(M, coarsest_n, nu[0], nu[1], omega, smoother).cycle(v, None, *gamma)
    dtype = torch.complex64 if prec == "c64" else torch.complex128
    for t in tunings:
        if t:
            helm.helm_set_tuning(h, t)
        z = helm.mg_precondition(h, to_gpu(v), dtype)
        assert rel_l2(to_np(z), ref) <= TOL[prec], t


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("smoother,nu,gamma", [("jacobi", (2, 2), (1, 1)), ("jacobi", (1, 2), (1, 3)),
                                               ("rb", (1, 1), (2, 2)), ("jacobi", (0, 1), (1, 1))])
@pytest.mark.parametrize("n,coarsest_n", [((65, 65), 17), ((81, 41), 17), ((41, 81), 11), ((43, 35), 21),
                                          ((17, 17, 17), 9), ((21, 13, 17), 6), ((13, 21, 33), 9)])
def test_fused_tail_any_cycle(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma):
    """The coarse tail on a thread-block cluster at every depth: lines and planes as rows, more
    blocks than rows, coarsest grids with an even number of rows, red-black and F / W cycles."""
    check_cycle(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma, [dict(tail_levels=t) for t in (-1, 2, 3, 4, 0)])


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("smoother,nu,gamma", [("jacobi", (1, 2), (1, 1)), ("jacobi", (2, 1), (1, 3)),
                                               ("jacobi", (2, 2), (2, 2)), ("rb", (1, 1), (1, 1)),
                                               ("rb", (2, 1), (1, 2)), ("rb", (1, 2), (1, 1)),
                                               ("jacobi", (3, 0), (1, 1)), ("rb", (0, 3), (1, 1))])
@pytest.mark.parametrize("n,coarsest_n", [((67, 35), 34), ((35, 67), 34), ((9, 5), 5), ((161, 97), 17), ((257, 193), 17)])
def test_2d_level_tiles(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma):
    """A level's way down and way up as one launch each: coarse interiors that fill the tiles exactly
    and that leave remainders, the smallest level, every tile shape, sweeps from zero and from a
    guess; more or fewer than one or two sweeps take the separate kernels."""
    check_cycle(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma, [dict(tail_levels=0)])


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("smoother,nu,gamma", [("jacobi", (1, 2), (1, 1)), ("rb", (1, 1), (1, 2)), ("rb", (2, 0), (1, 1))])
@pytest.mark.parametrize("n,coarsest_n", [((33, 17, 65), 9), ((17, 65, 33), 9), ((65, 33, 25), 9)])
def test_3d_level_kernels(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma):
    """The 3D sweeps (omega / D formed once in complex128), red-black from zero and from a guess, with
    chunks of one to eight planes."""
    check_cycle(helm, oracle, n, coarsest_n, prec, smoother, nu, gamma, [dict(tail_levels=0)])


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("nu,gamma,tail", [((1, 1), (1, 1), 0), ((2, 1), (1, 2), 0), ((1, 1), (2, 2), -1)])
@pytest.mark.parametrize("n,coarsest_n", [((33, 17, 65), 9), ((41, 73, 25), 10), ((97, 65), 17)])
def test_red_black_with_omega_one(helm, oracle, n, coarsest_n, prec, nu, gamma, tail):
    """omega = 1: the second colour's residuals are zero and the restriction takes only the first
    colour's, after the first sweep from zero (no diagonal term) and after later ones."""
    check_cycle(helm, oracle, n, coarsest_n, prec, "rb", nu, gamma, [dict(tail_levels=tail)], omega=1.0)


@pytest.mark.parametrize("n,coarsest_n", [((65, 33), 17), ((33, 17, 25), 9)])
@pytest.mark.parametrize("smoother", ["jacobi", "rb"])
def test_real_coefficients_outside_the_layers(helm, oracle, n, coarsest_n, smoother):
    """The shifted Laplacian keeps the widths, so its coefficients are real outside the layers and
    each axis takes the short form there: levels, tail, and the operator itself."""
    check_cycle(helm, oracle, n, coarsest_n, "c128", smoother, (1, 1), (1, 2), [dict(tail_levels=-1), dict(tail_levels=0)],
                pc="csl")
    P = problem(n, coarsest_n)
    h = gpu_handle(helm, P, pc="csl", prec="c128")
    A, M = oracle_pair(oracle, P, pc="csl")
    x = W.random_field(tuple(reversed(n)), 52)
    for which, op in (("A", A), ("M", M)):
        assert rel_l2(to_np(helm.helm_apply(h, to_gpu(x), which=which)), op.apply(x)) <= 1e-14


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [(33, 17, 25), (65, 57, 73), (81, 73, 81)])
def test_3d_apply_chunks(helm, oracle, n, prec):
    """The 3D operator with chunks of one, four and eight planes per thread and a last chunk that is
    not full.  complex128: 1e-14 as elsewhere; complex64: some 16 roundings of 6e-8 a node."""
    P = problem(n, 10)
    h = gpu_handle(helm, P, prec=prec)
    A, _ = oracle_pair(oracle, P)
    x = W.random_field(tuple(reversed(n)), 53)
    v = to_gpu(x)
    if prec == "c64":
        v = v.to(torch.complex64)
    assert rel_l2(to_np(helm.helm_apply(h, v)), A.apply(x)) <= (1e-6 if prec == "c64" else 1e-14)
