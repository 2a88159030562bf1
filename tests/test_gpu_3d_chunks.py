"""The 3D kernels with several planes per thread, against the oracle: grids large enough that the rule by
level size gives 2, 4, 8 and 16 planes, each with a last chunk that is not full.  Bounds as for the other
kernels of a cycle (1e-12 in complex128, 2e-5 in complex64) and of the operator (1e-14; complex64: some
16 roundings of 6e-8 a node)."""
import re

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


def problem(n):
    k2 = W.k2_well_growth(3, max(n), kh_max=0.5)[tuple(slice(0, m) for m in reversed(n))]
    return W.Problem("chunks", 3, list(n), np.ascontiguousarray(k2), np.zeros(tuple(reversed(n)), complex), coarsest_n=9)


def kernel_names(fn):
    """Names of the CUDA kernels fn launches (torch's profiler); empty when it records none."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    return {e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA}


# finest level, planes per thread of the sweep / the red-black sweep / the restriction:
# 2 / 1 / 1, 4 / 2 / 2, 8 / 4 / 4 and 16 / 8 / 8
@pytest.mark.parametrize("n,planes,smoother,nu,omega", [
    ((129, 129, 49), 2, "jacobi", (2, 1), 0.8),
    ((193, 129, 97), 4, "jacobi", (2, 1), 0.8),
    ((193, 129, 97), 4, "rb", (1, 1), 1.0),
    ((257, 129, 97), 8, "jacobi", (1, 2), 0.8),
    ((257, 257, 97), 16, "jacobi", (2, 1), 0.8),
    ((257, 257, 97), 16, "rb", (1, 1), 0.8),
    ((257, 257, 97), 16, "rb", (1, 1), 1.0),
])
def test_cycle_with_several_planes_per_thread(helm, oracle, n, planes, smoother, nu, omega):
    """One cycle from zero in either precision: the sweeps, the restriction (its shared planes are used more
    than once from six coarse planes a block on) and the prolongation; repeats are equal bit for bit."""
    P = problem(n)
    A, M = oracle_pair(oracle, P)
    v = W.random_field(tuple(reversed(n)), 51)
    ref = oracle.MG(M, 9, nu[0], nu[1], omega, smoother).cycle(v)
    vg = to_gpu(v)
    for prec, dtype in (("c64", torch.complex64), ("c128", torch.complex128)):
        h = gpu_handle(helm, P, prec=prec, smoother=smoother, nu=nu, omega=omega)
        z = helm.mg_precondition(h, vg, dtype)
        assert rel_l2(to_np(z), ref) <= TOL[prec], prec
        for _ in range(3):
            assert torch.equal(helm.mg_precondition(h, vg, dtype), z), prec
        if smoother == "jacobi":
            names = kernel_names(lambda: helm.mg_precondition(h, vg, dtype))
            assert not names or any(re.search(r"k_jacobi3<[^>]*\b%d>" % planes, s) for s in names), sorted(names)


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_apply_with_eight_planes_per_thread(helm, oracle, prec):
    n = (257, 257, 65)
    P = problem(n)
    h = gpu_handle(helm, P, prec=prec)
    A, _ = oracle_pair(oracle, P)
    x = W.random_field(tuple(reversed(n)), 53)
    v = to_gpu(x)
    if prec == "c64":
        v = v.to(torch.complex64)
    assert rel_l2(to_np(helm.helm_apply(h, v)), A.apply(x)) <= (1e-6 if prec == "c64" else 1e-14)
