"""Routes that a call may take without its results depending on it, compared bit
for bit:
  * blocks whose target pixels are all known are copied without iterating,
    unless the selected indices are asked for: an image with and without them;
  * blocks of one warp with different iteration counts and DC phases, and
    partly filled warps: a batch against its images alone;
  * the re-use form in one launch against its wavefront launches (taken while
    the stream is being captured)."""
import numpy as np
import pytest

from paper_2202_13926_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SB = [(32, 2), (32, 4), (32, 8), (32, 16), (24, 4), (24, 8), (16, 2), (16, 4), (16, 8), (8, 2), (8, 4), (4, 2), (4, 4)]


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


def _dev(img, mask):
    return torch.from_numpy(img).cuda(), torch.from_numpy(mask).cuda()


@pytest.mark.parametrize("S,B", SB)
@pytest.mark.parametrize("H,W", [(5, 3), (70, 90), (113, 251)])   # below and above the line of the small-launch kernel
@pytest.mark.parametrize("mask_kind", ["macroblock", "few_lost", "all_known", "none_known"])
def test_known_targets_are_copied(handle, S, B, H, W, mask_kind):
    mask = {"macroblock": synth.macroblock_mask(H, W, 3, 0.2), "few_lost": synth.iid_mask(H, W, 4, 0.02),
            "all_known": np.ones((H, W), np.uint8), "none_known": np.zeros((H, W), np.uint8)}[mask_kind]
    t, m = _dev(synth.sinusoid_image(H, W, 5), mask)
    kw = dict(block=B, border=(S - B) // 2, iters=25)
    n = -(-H // B) * -(-W // B)
    seq = torch.zeros(n * 25, dtype=torch.int16, device="cuda")
    from paper_2202_13926_gb300 import fsr
    opts = [{}]
    if S == 32:
        opts += [dict(reuse=0.5)] + ([dict(update="conj_pair")] if B == 4 else [])
    for o in opts:
        full = handle.reconstruct(t, m, seq_out=seq, **kw, **o).clone()
        empty = fsr.fsr_empty_blocks(handle.ptr)
        got = handle.reconstruct(t, m, out=torch.full_like(t, -9.0), **kw, **o)
        assert torch.equal(got, full)
        assert fsr.fsr_empty_blocks(handle.ptr) == empty


@pytest.mark.parametrize("S,B", [(16, 4), (8, 2), (8, 4), (4, 2), (4, 4)])
def test_blocks_of_a_warp_do_not_meet(handle, S, B):
    from paper_2202_13926_gb300 import fsr
    sizes = [(B, B), (B, 3 * B), (33, 29), (64, 80), (B, 33 * B)]
    iters = [40, 1, 17, 33, 0]
    ims = []
    for i, (H, W) in enumerate(sizes):
        img = synth.sinusoid_image(H, W, i)
        img[: H // 2] = 90.0   # flat: blocks that stay in the DC phase beside others
        ims.append(_dev(img, synth.iid_mask(H, W, 20 + i, 0.5)))
    outs = [torch.zeros_like(a) for a, _ in ims]
    p = fsr.make_params(block=B, border=(S - B) // 2)
    fsr.fsr_reconstruct_batch(handle.ptr, [fsr.image_desc(a, m, o, k) for (a, m), o, k in zip(ims, outs, iters)], p)
    for (a, m), o, k in zip(ims, outs, iters):
        assert torch.equal(o, handle.reconstruct(a, m, block=B, border=(S - B) // 2, iters=k))


@pytest.mark.parametrize("B", [2, 4, 8, 16])
def test_reuse_rows_equal_wavefronts(handle, B):
    from paper_2202_13926_gb300 import fsr
    sizes = [(B, B), (50, 7), (7, 70), (61, 83)]   # one block, one column, one row, ragged
    ims = [_dev(synth.sinusoid_image(H, W, i), synth.iid_mask(H, W, 9 + i, 0.6)) for i, (H, W) in enumerate(sizes)]
    kw = dict(block=B, border=(32 - B) // 2, iters=20, reuse=0.5)
    p = fsr.make_params(**kw)
    rows = [torch.zeros_like(a) for a, _ in ims]
    fsr.fsr_reconstruct_batch(handle.ptr, [fsr.image_desc(a, m, o, 20) for (a, m), o in zip(ims, rows)], p)
    handle.check_status()
    waves = [torch.zeros_like(a) for a, _ in ims]
    d = [fsr.image_desc(a, m, o, 20) for (a, m), o in zip(ims, waves)]
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        fsr.fsr_reconstruct_batch(handle.ptr, d, p)
    g.replay()
    torch.cuda.synchronize()
    for r, w, (a, m) in zip(rows, waves, ims):
        assert torch.equal(r, w)
        assert torch.equal(r, handle.reconstruct(a, m, **kw))
