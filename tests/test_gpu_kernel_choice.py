"""Which build of the FP64 kernel a launch runs (csrc/tt_kernel64.cu launch64): the
one without a register cap where every ray has a lane of its own, for one camera
and for a batch alike, else the one that fits three blocks on an SM.  The kernels
launched are listed by the profiler."""
import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def kernels(call):
    """Names of the tracing kernels that a call launches."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):          # (the first profile of a process may miss what it starts up with)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
    return [e.name for e in prof.events() if "trace_kernel" in e.name]


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
