"""The re-use form in one launch: the waits of its block rows for one another.
They end by themselves whatever the images' sizes and iteration counts, and one
that cannot end gives up, is reported, and leaves the handle usable."""
import pytest

from paper_2202_13926_gb300 import synth

gpu = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2202_13926_gb300 import fsr
    h = fsr.Handle(0)
    yield h
    h.close()


def _image(H, W, seed):
    return (torch.from_numpy(synth.sinusoid_image(H, W, seed)).cuda(),
            torch.from_numpy(synth.iid_mask(H, W, seed, 0.6)).cuda())


@gpu
def test_a_row_may_stand_still_behind_many_others(handle):
    """Twelve images that are done at once and a tall narrow one, whose rows then
    occupy the whole launch: 300 of its rows of two blocks start one after
    another (over 10 ms at K = 100), each watching a row that has not begun.  The
    base limit is 2 ms; a block takes 0.02 ms, so blocks keep finishing."""
    from paper_2202_13926_gb300 import fsr
    shapes = [(108, 480, 1)] * 12 + [(4000, 8, 100)]
    ims = [_image(H, W, i) for i, (H, W, _) in enumerate(shapes)]
    outs = [torch.full_like(a, -9.0) for a, _ in ims]
    d = [fsr.image_desc(a, m, o, k) for (a, m), o, (_, _, k) in zip(ims, outs, shapes)]
    fsr.fsr_inject_row_wait_fault(handle.ptr, base_ns=2_000_000)
    fsr.fsr_reconstruct_batch(handle.ptr, d, fsr.make_params(reuse=0.5))
    handle.check_status()
    for (a, m), o, (_, _, k) in zip(ims, outs, shapes):
        assert torch.equal(o, handle.reconstruct(a, m, iters=k, reuse=0.5))
    handle.check_status()


@gpu
def test_row_wait_timeout_is_reported_and_the_handle_recovers(handle):
    from paper_2202_13926_gb300 import fsr
    t, m = _image(64, 96, 3)
    good = handle.reconstruct(t, m, iters=20, reuse=0.5)
    handle.check_status()
    fsr.fsr_inject_row_wait_fault(handle.ptr, base_ns=20_000_000, skip_first_row=True)
    out = torch.full_like(t, -9.0)
    fsr.fsr_reconstruct(handle.ptr, t, m, fsr.make_params(iters=20, reuse=0.5), out)
    with pytest.raises(fsr.FsrError) as e:
        handle.check_status()
    assert e.value.code == fsr.FSR_ERR_TIMEOUT
    assert "block row" in str(e.value)
    assert torch.all(out == -9.0)             # no row has the one above it
    handle.check_status()                     # the word was cleared
    again = handle.reconstruct(t, m, iters=20, reuse=0.5)
    handle.check_status()
    assert torch.equal(again, good)


def _constant(name):
    import os
    import re
    from paper_2202_13926_gb300 import build
    text = "".join(open(os.path.join(build.CSRC, f)).read() for f in ("fsr_launch.h", "fsr_coop.cuh", "fsr_reuse.cuh",
                                                                       "fsr_internal.h"))
    return int(re.search(rf"constexpr int {name} = (\d+);", text).group(1))


def _random(H, W, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return (torch.rand(H, W, device="cuda", generator=g) * 255,
            (torch.rand(H, W, device="cuda", generator=g) >= 0.6).to(torch.uint8))


@gpu
@pytest.mark.parametrize("B", [2, 4, 8, 16])
@pytest.mark.parametrize("wider", [False, True])
def test_wide_wavefronts_equal_single_images(handle, B, wider):
    """Batches whose wavefronts hold more blocks than the CTA-per-block kernels
    take (the one-warp kernel in CTAs of 4 warps, and of 8 beyond one wave of
    those): every image is that of its own call, which runs in one launch."""
    from paper_2202_13926_gb300 import fsr
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lag = -(-((32 - B) // 2) // B) + 1
    least = _constant("kCoopReusePerSm") * sms
    four = _constant("kCtasPerSmReuse") * _constant("kWarpsReuse") * sms
    rows = 64
    n = (four if wider else least) // rows + 2
    assert n <= 48 and n * rows > least and (n * rows > four) == wider
    assert n * rows > _constant("kCoopRowsPerSm") * sms
    H, W = rows * B - 1, (lag * rows + 3) * B - 1   # wavefronts of `rows` blocks per image
    ims = [_random(H, W, i) for i in range(3)]
    outs = [torch.full_like(ims[0][0], -9.0) for _ in range(n)]
    kw = dict(block=B, border=(32 - B) // 2, reuse=0.5)
    fsr.fsr_reconstruct_batch(handle.ptr, [fsr.image_desc(*ims[i % 3], o, 3) for i, o in enumerate(outs)],
                              fsr.make_params(**kw))
    one = [handle.reconstruct(t, m, iters=3, **kw) for t, m in ims]
    handle.check_status()
    for i, o in enumerate(outs):
        assert torch.equal(o, one[i % 3]), i


@gpu
@pytest.mark.parametrize("B,W", [(4, 24), (16, 40)])
def test_more_rows_than_the_progress_ring_holds(handle, B, W):
    """A tall image: a row takes over the slot of a row kRowRing before it.
    Against the wavefront launches (taken while the stream is being captured)."""
    from paper_2202_13926_gb300 import fsr
    H = (_constant("kRowRing") + 70) * B - 1
    t, m = _random(H, W, B)
    p = fsr.make_params(block=B, border=(32 - B) // 2, iters=3, reuse=0.5)
    out, ref = torch.full_like(t, -9.0), torch.full_like(t, -9.0)
    fsr.fsr_reconstruct(handle.ptr, t, m, p, out)
    handle.check_status()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        fsr.fsr_reconstruct(handle.ptr, t, m, p, ref)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


@gpu
def test_more_rows_than_the_progress_ring_holds_in_a_batch(handle):
    """Rows of one image take over slots of others with other iteration counts."""
    from paper_2202_13926_gb300 import fsr
    shapes = [(108, 200, 1 + 20 * (i % 2)) for i in range(39)] + [(4300, 24, 9)]
    assert sum(-(-h // 4) for h, _, _ in shapes) > _constant("kRowRing")
    ims = [_random(h, w, i) for i, (h, w, _) in enumerate(shapes)]
    outs = [torch.full_like(t, -9.0) for t, _ in ims]
    d = [fsr.image_desc(t, m, o, k) for (t, m), o, (_, _, k) in zip(ims, outs, shapes)]
    fsr.fsr_reconstruct_batch(handle.ptr, d, fsr.make_params(reuse=0.5))
    for (t, m), o, (_, _, k) in zip(ims, outs, shapes):
        assert torch.equal(o, handle.reconstruct(t, m, iters=k, reuse=0.5))
    handle.check_status()


@gpu
def test_progress_rings_are_used_again_while_calls_are_in_flight(handle):
    """More calls on three streams than the handle has rings."""
    from paper_2202_13926_gb300 import fsr
    ims = [_random(61 + 8 * i, 83 - 9 * i, i) for i in range(4)]
    alone = [handle.reconstruct(t, m, iters=15, reuse=0.5) for t, m in ims]
    n = 5 * _constant("kRowSlots") + 3
    outs = [torch.full_like(ims[j % 4][0], -9.0) for j in range(n)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    p = fsr.make_params(iters=15, reuse=0.5)
    torch.cuda.synchronize()
    for j, o in enumerate(outs):
        fsr.fsr_reconstruct(handle.ptr, *ims[j % 4], p, o, streams[j % 3])
    torch.cuda.synchronize()
    handle.check_status()
    for j, o in enumerate(outs):
        assert torch.equal(o, alone[j % 4]), j


def test_row_wait_hook_rejects_bad_arguments():
    from paper_2202_13926_gb300 import build, fsr
    build.build()
    assert fsr.load_library().fsr_inject_row_wait_fault(None, 0, 0) == fsr.FSR_ERR_INVALID_ARG
