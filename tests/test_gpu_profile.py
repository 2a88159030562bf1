"""Launch timing counts every pass of a solve: the vector passes of Bi-CGSTAB, which also form its inner products,
and the passes that round a vector for the complex64 cycle on the way."""
import numpy as np
import pytest

from helpers import gpu_handle, to_gpu
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


def problem(n):
    return W.Problem("profile", 2, n, W.k2_well_growth(2, n, kh_max=0.3), W.gaussian_source(2, n, 0.1, 3), coarsest_n=17)


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_bicgstab_passes_are_timed(helm, prec):
    """Five vector passes an iteration (four and the last update when it ends in the middle): bytes per
    node 64 + 32 + 48 + 32 + 96 and the cycles' vectors, 8 or 16 bytes each."""
    P = problem(129)
    h = gpu_handle(helm, P, prec=prec)
    f = to_gpu(P.f)
    helm.helm_profile(h, True)
    x, st = helm.krylov_solve(h, f, tol=1e-8, method="bicgstab", maxit=200)
    v = helm.helm_profile_read(h)["vector"]
    helm.helm_profile(h, False)
    its, node = st.iterations, 129 * 129
    assert its >= 3
    assert v["launches"] >= 5 * its - 1
    per = 272 + (2 * 8 + 2 * 8 if prec == "c64" else 2 * 16)  # rounded copies of p and s, or none; y and z
    assert v["bytes"] >= node * per * (its - 1)
    assert np.isfinite(v["ms"]) and v["ms"] > 0


def test_rounding_on_the_way_is_counted(helm):
    """The first launch of a complex64 cycle reads the complex128 vector (16 bytes a node) and writes the rounded
    one beside what it moves otherwise: 42 instead of 26 bytes a node, then 34 for the way up."""
    P = problem(257)
    h = gpu_handle(helm, P, prec="c64")
    v = to_gpu(P.f)
    helm.helm_profile(h, True)
    helm.mg_precondition(h, v)
    fine = helm.helm_profile_read(h)["smooth_fine"]
    helm.helm_profile(h, False)
    assert fine["launches"] == 2
    assert abs(fine["bytes"] / 255 ** 2 - 76) < 1e-9
