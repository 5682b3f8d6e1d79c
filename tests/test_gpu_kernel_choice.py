"""Which build of the FP64 kernel a launch runs (csrc/tt_kernel64.cu launch64): the
one without a register cap where every ray has a lane of its own, for one camera
and for a batch alike, else the one that fits three blocks on an SM.  The kernels
launched are listed by the profiler."""
import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def kernels(call):
    """Names of the tracing kernels that a call launches (skips where the profiler does
    not list even a kernel of torch's own)."""
    from torch.profiler import ProfilerActivity, profile
    marker = torch.zeros(1, device="cuda")
    for _ in range(2):          # (the first profile of a process may miss what it starts up with)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            marker.add_(1.0)
            call()
            torch.cuda.synchronize()
    names = [e.name for e in prof.events()]
    if not any("elementwise" in n for n in names):
        pytest.skip("the profiler lists no kernels here")
    return [n for n in names if "trace_kernel" in n]


@pytest.mark.parametrize("images,side,few", [(1, 16, True), (3, 16, True), (65, 8, True), (1, 256, False), (4, 128, False)])
def test_build_by_number_of_rays(images, side, few):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus as T
    imgs = [scenes.kerr_disk(side).replace(a=0.01 * k, rtol=1e-6, atol=1e-6) for k in range(images)]
    outs = [T.alloc_outputs(s.npix) for s in imgs]
    call = (lambda: T.trace(imgs[0], out=outs[0])) if images == 1 else (lambda: T.trace_batch(imgs, outs))
    rays = sum(s.npix for s in imgs)
    assert few == (rays <= 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count)
    names = kernels(call)
    assert len(names) == (images + 63) // 64, names
    for n in names:
        assert ("trace_kernel64<" in n) == few and ("regcap" in n) == (not few), names


@pytest.mark.parametrize("precision,band,each", [(scenes.FP64, 0.0, 1), (scenes.DOUBLE_FLOAT, 0.0, 1),
                                                 (scenes.MIXED, 0.0, 2), (scenes.MIXED_PAIR, 0.0, 2),
                                                 (scenes.MIXED_PAIR, -1.0, 1), (scenes.MIXED_SPLIT, 0.0, 1),
                                                 (scenes.MIXED_SPLIT, 0.15, 2)])
def test_launch_count_counts_kernels(precision, band, each):
    """The near-critical rays of the mixed paths run in a kernel of their own, which
    tartarus_launch_count and a graph's launches_per_replay count too."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus as T
    sc = scenes.kerr_disk(24, precision).replace(rtol=1e-7, atol=1e-7, critical_band=band)
    out = T.alloc_outputs(sc.npix)
    n0 = T.launch_count()
    T.trace(sc, out=out)
    assert T.launch_count() - n0 == each
    assert len(kernels(lambda: T.trace(sc, out=out))) == each
    imgs = [sc] * 65
    outs = [T.alloc_outputs(sc.npix) for _ in imgs]
    n0 = T.launch_count()
    status = []
    T.trace_batch_noalloc(imgs, outs, status_out=status)
    assert T.launch_count() - n0 == 2 * each and status == [0] * 65
    assert T.TraceGraph(imgs, outs).launches_per_replay == 2 * each
    torch.cuda.synchronize()


@pytest.mark.parametrize("method", [scenes.DOPRI5, scenes.CASH_KARP, scenes.GBS])
@pytest.mark.parametrize("side", [16, 256])
def test_benchmark_names_the_kernel(method, side):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import bench
    from paper_2609_08989_gb300 import tartarus as T
    sc = scenes.kerr_disk(side).replace(method=method, rtol=1e-6, atol=1e-6)
    out = T.alloc_outputs(sc.npix)
    names = kernels(lambda: T.trace(sc, out=out))
    assert len(names) == 1 and bench.kernel_name(sc) in names[0].replace(" ", ""), (names, bench.kernel_name(sc))
