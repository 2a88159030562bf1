"""What the set-up calls leave behind: work in flight, memory, and the kernels that the cycles run."""
import re

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


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_complex64_handles_hold_no_complex128_diagonals(helm):
    """omega / D in complex128 (16 bytes a node) belongs to complex128 cycles: a complex64 handle forms it in
    its first one, a complex128 handle at creation."""
    n = (97, 97, 97)
    v = to_gpu(W.random_field(n, 61))
    z = torch.zeros_like(v)  # what mg_precondition allocates for its result is then in torch's cache
    del z
    taken = {}
    for prec in ("c64", "c128"):
        h = handle(helm, n, prec=prec)
        drops = []
        for _ in range(2):
            before = free_bytes()
            z = helm.mg_precondition(h, v, torch.complex128)
            drops.append(before - free_bytes())
            del z
        taken[prec] = drops
    assert taken["c64"][0] >= 15 * 97 ** 3 and taken["c64"][1] == 0
    assert taken["c128"] == [0, 0]


@pytest.mark.parametrize("n", [(65, 65), (33, 33, 33)])
def test_complex128_cycles_on_a_complex64_handle(helm, n):
    """They equal those of a complex128 handle bit for bit, leave the complex64 cycles as they were, and the
    first of them can be inside a stream capture."""
    v = to_gpu(W.random_field(tuple(reversed(n)), 62))
    ref = helm.mg_precondition(handle(helm, n, prec="c128", nu=(1, 2)), v, torch.complex128)
    for tail in (-1, 0):
        h = handle(helm, n, prec="c64", nu=(1, 2))
        helm.helm_set_tuning(h, dict(tail_levels=tail))
        z64 = helm.mg_precondition(h, v)
        z = helm.mg_precondition(h, v, torch.complex128)
        if tail == -1:
            assert torch.equal(z, ref)
        assert float(torch.linalg.vector_norm(z - ref) / torch.linalg.vector_norm(ref)) <= 1e-12
        assert torch.equal(helm.mg_precondition(h, v), z64)
    # captured first, then run
    s = torch.cuda.Stream()
    h = handle(helm, n, stream=s, prec="c64", nu=(1, 2))
    x = torch.zeros_like(v)
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        helm.mg_vcycle(h, v, x)
    g.replay()
    torch.cuda.synchronize()
    y = torch.zeros_like(v)
    helm.mg_vcycle(h, v, y)
    torch.cuda.synchronize()
    assert float(x.abs().max()) > 0 and torch.equal(x, y)


def test_noalloc_in_complex128_on_a_complex64_handle(helm):
    """The allocation-free entry point takes no memory there either, gives helm_mg_conv's result and leaves the
    complex64 cycles as they were."""
    n = (257, 257)
    v = to_gpu(W.random_field(n, 63))
    warm = handle(helm, n, prec="c64")
    helm.helm_mg_conv_noalloc(warm, v, torch.zeros_like(v), maxcyc=2)
    h = handle(helm, n, prec="c64")
    z64 = helm.mg_precondition(h, v)
    x = torch.zeros_like(v)
    before = free_bytes()
    cycles, factor = helm.helm_mg_conv_noalloc(h, v, x, tol=1e-6, maxcyc=30)
    assert free_bytes() >= before
    assert torch.equal(helm.mg_precondition(h, v), z64)
    xr, cr, fr = helm.helm_mg_conv(h, v, tol=1e-6, maxcyc=30)
    assert cycles == cr and torch.equal(x, xr)
    assert torch.equal(helm.mg_precondition(h, v), z64)


def kernel_names(fn):
    """Names of the CUDA kernels fn launches (torch's profiler); None when it records none."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    return {e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA} or None


@pytest.mark.parametrize("change", ["round trip", "tail only", "autotuned in complex128"])
def test_tiles_by_size_survive(helm, change):
    """Reading a handle's tuning and setting it again, changing another field of it, or autotuning the
    complex128 cycle (which has no such tiles) leaves the complex64 cycle on the tiles that suit its levels."""
    h = handle(helm, (513, 513), prec="c64")
    v = to_gpu(W.random_field((513, 513), 64))

    def tiles():
        names = kernel_names(lambda: helm.mg_precondition(h, v))
        return names and set(re.findall(r"k_(?:pre2_restrict|prolong_post2)<[^>]*>", " ".join(sorted(names))))

    tiles()  # the first profile of a process may record nothing
    before, z = tiles(), helm.mg_precondition(h, v)
    reported = helm.helm_get_tuning(h)
    if change == "round trip":
        helm.helm_set_tuning(h, reported)
    elif change == "tail only":
        helm.helm_set_tuning(h, dict(tail_levels=reported["tail_levels"]))
    else:
        tuning, _ = helm.helm_autotune(h, "c128", reps=2)
        assert tuning == helm.helm_get_tuning(h) and tuning["level_tile"] == reported["level_tile"]
        helm.helm_set_tuning(h, dict(tail_levels=reported["tail_levels"]))
    assert helm.helm_get_tuning(h)["level_tile"] == reported["level_tile"]
    after = tiles()
    assert before is None or after is None or (after == before and len(before) >= 4)
    assert torch.equal(helm.mg_precondition(h, v), z)
