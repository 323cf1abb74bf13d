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


def test_row_wait_hook_rejects_bad_arguments():
    from paper_2202_13926_gb300 import build, fsr
    build.build()
    assert fsr.load_library().fsr_inject_row_wait_fault(None, 0, 0) == fsr.FSR_ERR_INVALID_ARG
