"""The CTA-per-block FP32 kernel (few blocks in a launch) against the one-warp
kernel: same arithmetic, so images, selected indices and empty-block counts
are equal bit for bit.  The one-warp kernel runs the same image when a second
image lifts the launch above the line."""
import numpy as np
import pytest

from paper_2202_13926_gb300 import synth

pytestmark = pytest.mark.gpu

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


# one block; ragged in both directions; at B = 4 on 152 SMs the last size of the
# four-warp form (456 blocks), the first and the last of the two-warp form (475,
# 1672) and the first of the one-warp kernel; two warps at the other B
SIZES = [(3, 2, 4), (33, 47, 2), (61, 83, 4), (76, 96, 4), (76, 97, 4), (152, 176, 4), (152, 177, 4), (97, 101, 8),
         (131, 90, 16), (50, 61, 2), (203, 239, 8), (399, 470, 16)]


@pytest.mark.parametrize("H,W,B", SIZES)
@pytest.mark.parametrize("mask_kind", ["iid", "sparse", "macroblock"])
@pytest.mark.parametrize("K,opts", [(0, {}), (1, {}), (60, {}), (40, dict(rho=0.83, gamma=0.3, freq_weight=False))])
def test_cta_per_block_equals_one_warp(handle, H, W, B, mask_kind, K, opts):
    from paper_2202_13926_gb300 import fsr
    dev = torch.device("cuda:0")
    img = synth.sinusoid_image(H, W, seed=H + W)
    mask = (synth.iid_mask(H, W, 5, 0.5) if mask_kind == "iid" else synth.iid_mask(H, W, 6, 0.998)
            if mask_kind == "sparse" else synth.macroblock_mask(H, W, 7, 0.5))
    t = torch.from_numpy(np.where(mask, img, np.nan).astype(np.float32)).to(dev)   # unknown values are not used
    m = torch.from_numpy(mask).to(dev)
    n = -(-H // B) * -(-W // B)
    border = (32 - B) // 2
    big = torch.zeros(512, 1280, device=dev)
    big_mask = torch.ones(512, 1280, dtype=torch.uint8, device=dev)

    def run(extra, batch):
        out = torch.full((H, W), -7.0, device=dev)
        seq = torch.full((n * max(K, 1),), -7, dtype=torch.int16, device=dev)
        p = fsr.make_params(block=B, border=border, iters=K, seq_out=None if batch else seq, **opts)
        if batch:
            d = [fsr.image_desc(t, m, out, K, seq)]
            if extra:   # K = 0: after this image in the work list
                d.append(fsr.image_desc(big, big_mask, torch.empty_like(big), 0))
            fsr.fsr_reconstruct_batch(handle.ptr, d, p)
        else:
            fsr.fsr_reconstruct(handle.ptr, t, m, p, out)
        return out, seq, fsr.fsr_empty_blocks(handle.ptr)

    ref = run(True, True)
    assert torch.isfinite(ref[0]).all()
    for got in (run(False, False), run(False, True)):
        assert torch.equal(got[0], ref[0])
        assert torch.equal(got[1], ref[1])
        assert got[2] == ref[2]
