"""FP64 handles on a device with little memory left: the memory of the digit-
splitting paths is optional, so a build or create that fits without it succeeds.

The device's free memory is taken by one plain allocation; the sizes below
leave some hundred MB.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MB = 1 << 20


def hog(leave):
    """All but `leave` bytes of the device's free memory."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def close(got, ref, tol):
    for x, r in zip(got, ref):
        assert np.linalg.norm(x - r) <= tol * np.linalg.norm(r)


def test_third_accumulator_does_not_fit(esmf):
    """Digit tiles and two accumulators do not fit together, two accumulators do."""
    import torch
    n, m = 800, 64
    w = W.small_random(n, 1, 3, tol=1e-6, edge=400.0)             # a thin gas: few bricks
    D = torch.randn((m, n, n), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    J, K = torch.empty_like(D), torch.empty_like(D)
    tiles = 100 * 100 * (6 * 2 * 16 * 128 + 32) + 50 * 101 * (6 * 16 * 128 + 32)
    acc = m * n * n * 8
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp64") as fb:
        fb.set_path("cuda_core")
        ref = [x.cpu().numpy() for x in fb.build(D[:2])[:2]]      # loads the kernels
        fb.set_path("auto")
        fb.build(D[:2])
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp64") as fb:
        fill = hog(2 * acc + tiles // 2)
        try:
            fb.build(D, J, K, want_traces=False)
            used = fb.stats()["device_bytes"]
            fb.build(D, J, K, want_traces=False)
            assert fb.stats()["device_bytes"] == used
        finally:
            del fill
            torch.cuda.empty_cache()
        close([x[:2].cpu().numpy() for x in (J, K)], ref, 1e-11)


def test_direct_budget(esmf):
    """A direct handle with the scratch buffer stays in its budget, digit tiles included."""
    import torch
    w = W.small_random(96, 1, 4, tol=1e-10)
    D = torch.from_numpy(w.D).cuda()
    acc = (3 * 96 * 96 + 1) * 8
    with esmf.FockBuilder(w.basis, w.tol, "direct", "fp64", budget_bytes=1 << 20) as fb:
        base = fb.stats()
    assert base["scratch_bytes"] == 0 and base["n_chunks"] == 0
    taken = 0
    for extra in range(0, 24 * MB, MB // 4):
        budget = base["device_bytes"] + extra
        with esmf.FockBuilder(w.basis, w.tol, "direct", "fp64", budget_bytes=budget) as fb:
            if fb.stats()["scratch_bytes"]:
                taken += 1
                fb.build(D)
                assert fb.stats()["device_bytes"] <= budget + acc
    assert taken > 10


def test_create_direct(esmf):
    """A direct handle is made whenever it fits without the scratch buffer."""
    import torch
    w = W.small_random(200, 2, 4, tol=1e-10, edge=10.0, min_dist=1.0)
    D = torch.from_numpy(w.D).cuda()

    def make():
        with esmf.FockBuilder(w.basis, w.tol, "direct", "fp64") as fb:
            return fb.stats()
    st = make()
    assert st["scratch_bytes"] > 500 * MB
    missed = 0
    for less in (64, 40, 20, 16, 12, 8, 6, 4, 2, 0):
        fill = hog(st["device_bytes"] + 80 * MB - less * MB)
        try:
            missed += make()["scratch_bytes"] == 0
        finally:
            del fill
    for less in range(0, 40, 2):                                  # without the slack of the loop above
        fill = hog(st["device_bytes"] + 8 * MB - less * MB)
        try:
            missed += make()["scratch_bytes"] == 0
        finally:
            del fill
            torch.cuda.empty_cache()
    assert missed > 0                                             # the fallback ran
    with esmf.FockBuilder(w.basis, 1e-4, "direct", "fp64") as fb:
        assert fb.device_error() == 0 and torch.isfinite(fb.build(D)[0]).all()


def test_staging_of_host_buffers_does_not_fit(esmf):
    """Memory that a build cannot do without takes the digit tiles' place."""
    import torch
    n, m = 800, 16
    w = W.small_random(n, 1, 3, tol=1e-6, edge=400.0)
    D = torch.randn((m, n, n), dtype=torch.float64, generator=torch.Generator().manual_seed(1)).pin_memory()
    pin = lambda: torch.empty((m, n, n), dtype=torch.float64).pin_memory()  # noqa: E731
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp64") as fb:
        ref = [x.numpy() for x in fb.build_host(D, pin(), pin())[:2]]
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp64") as fb:
        one = torch.zeros((1, n, n), dtype=torch.float64, device="cuda")
        fb.build(one)
        fill = hog(4 * m * n * n * 8 - 64 * MB)                   # less than the staging alone
        try:
            got = [x.numpy() for x in fb.build_host(D, pin(), pin())[:2]]
        finally:
            del fill
            torch.cuda.empty_cache()
        close(got, ref, 1e-11)


def test_density_tiles_do_not_fit(esmf):
    """A density-fitted handle goes back to cuBLAS when the tiles of many densities do not fit."""
    import torch
    n, m = 130, 512
    w = W.small_random(n, 1, 6, edge=12.0, min_dist=1.0)
    aux = W.even_tempered_aux(w.basis, count=2)
    D = torch.randn((m, n, n), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    J, K = torch.empty_like(D), torch.empty_like(D)
    with esmf.FockBuilder(w.basis, 0.0, "df", "fp64", aux=aux) as fb:
        ref = [x.cpu().numpy() for x in fb.build(D[:2])[:2]]
        fb.build(D, J, K, want_traces=False)                      # loads cuBLAS' kernels for these sizes
    with esmf.FockBuilder(w.basis, 0.0, "df", "fp64", aux=aux) as fb:
        fb.build(D[:1])
        tiles = m * 6 * 114688                                    # 128 x 64 tiles of 112 KB, two by three a density
        fill = hog(tiles - 16 * MB)
        try:
            fb.build(D, J, K, want_traces=False)
            st = fb.stats()["store_bytes"]
        finally:
            del fill
            torch.cuda.empty_cache()
        assert st == 2 * len(aux[1]) * n * n * 8
        close([x[:2].cpu().numpy() for x in (J, K)], ref, 1e-12)
        fb.build(D, J, K, want_traces=False)
        close([x[:2].cpu().numpy() for x in (J, K)], ref, 1e-12)


def test_captured_builds_keep_their_memory(esmf):
    """A graph replays over the memory that it was captured with: none of it goes back for another call."""
    import torch
    n, m = 800, 16
    w = W.small_random(n, 1, 3, tol=1e-6, edge=400.0)
    D = torch.randn((m, n, n), dtype=torch.float64, generator=torch.Generator().manual_seed(1)).pin_memory()
    J, K = torch.empty_like(D).pin_memory(), torch.empty_like(D).pin_memory()
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp64") as fb:
        one = D[:1].cuda()
        Jd, Kd = torch.empty_like(one), torch.empty_like(one)
        fb.build(one, Jd, Kd, want_traces=False)
        ref = [x.cpu().numpy() for x in (Jd, Kd)]
        graph = torch.cuda.CUDAGraph()
        stream = torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            fb.build(one, Jd, Kd, want_traces=False, stream=stream)
        used = fb.stats()["device_bytes"]
        fill = hog(4 * m * n * n * 8 - 64 * MB)
        try:
            with pytest.raises(esmf.EsmfError, match="out of memory"):
                fb.build_host(D, J, K)
        finally:
            del fill
            torch.cuda.empty_cache()
        assert fb.stats()["device_bytes"] >= used
        Jd.zero_(), Kd.zero_()
        graph.replay()
        torch.cuda.synchronize()
        close([x.cpu().numpy() for x in (Jd, Kd)], ref, 1e-11)
