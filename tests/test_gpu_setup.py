"""What the set-up calls leave behind: work in flight, memory, and the kernels that the cycles run."""
import numpy as np
import pytest

from helpers import mg_params, to_gpu
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


def handle(helm, n, stream=None, **kw):
    dim = len(n)
    k2 = W.k2_well_growth(dim, max(n), kh_max=0.5)[tuple(slice(0, m) for m in reversed(n))]
    return helm.helm_create(dim, n, torch.from_numpy(np.ascontiguousarray(k2)).cuda(), stream=stream,
                            mg=mg_params(helm, coarsest_n=9, **kw))


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_set_tuning_waits_for_the_tail_images(helm, prec):
    """A tail copies its prebuilt image before it waits for the kernel ahead of it, so that kernel must not
    be the one that builds the image: with the handle's stream kept busy, helm_set_tuning returns only
    once a new image is in memory."""
    s = torch.cuda.Stream()
    h = handle(helm, (65, 65), stream=s, prec=prec)
    for levels in (2, 3):
        s.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(100_000_000)  # about 50 ms
        helm.helm_set_tuning(h, dict(tail_levels=levels))
        assert s.query(), levels
