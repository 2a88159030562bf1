"""FGMRES at the ends of its range of restart lengths, with every arithmetic of the Arnoldi process: whole cycles
of 1, 2, 63 and 64 steps (without a preconditioner, so that the solve needs several)."""
import numpy as np
import pytest

from helpers import gpu_handle, oracle_pair, to_gpu, to_np
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


@pytest.mark.parametrize("restart", [1, 2, 63, 64])
@pytest.mark.parametrize("gs", ["fp64", "df", "dcgs2"])
def test_whole_cycles(helm, oracle, restart, gs):
    """Two whole cycles and a third run, and the reported residual is that of the solution."""
    P = W.Problem("restart", 2, 33, W.k2_well_growth(2, 33, kh_max=0.3), W.random_box_source(2, 33, 5), coarsest_n=17)
    A, _ = oracle_pair(oracle, P)
    h = gpu_handle(helm, P, pc="none", gs=gs)
    x, st = helm.krylov_solve(h, to_gpu(P.f), tol=1e-8, restart=restart, maxit=3 * restart, history=True, raise_on_noconv=False)
    assert st.status in (helm.HELM_OK, helm.HELM_ERR_NOCONV) and len(st.history) == st.iterations >= 2 * restart
    true = np.linalg.norm(P.f - A.apply(to_np(x))) / np.linalg.norm(P.f)
    assert abs(true - st.rel_res) <= 1e-9
