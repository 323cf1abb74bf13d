"""Launches of more blocks than the CTA-per-block kernel takes (kCoopBlocksPerSm
per SM, read from its source so that a later move of the line moves the sizes):
the one-warp FP32 kernel of S = 32 at every B."""
import os
import re

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


def wide_size(B, over=1.05):
    """Ragged (H, W) of `over` times the blocks of the line."""
    from paper_2202_13926_gb300 import build
    text = open(os.path.join(build.CSRC, "fsr_launch.h")).read()
    line = int(re.search(r"kCoopBlocksPerSm = (\d+);", text).group(1))
    blocks = over * line * torch.cuda.get_device_properties(0).multi_processor_count
    n = int(blocks ** 0.5) + 1
    return n * B - 1, (n + 1) * B - (B // 2)


@pytest.mark.parametrize("B", [2, 4, 8, 16])
@pytest.mark.parametrize("over", [1.05, 8.0])   # one entry at a time; takes of several entries
@pytest.mark.parametrize("kind", ["macroblock", "few_lost", "half_lost", "all_known"])
def test_known_targets_are_copied(handle, B, over, kind):
    """An image whose blocks are all iterated (selected indices asked for)
    against the call that copies the blocks without an unknown pixel."""
    if B >= 8 and over > 2:
        over = 3.0
    H, W = wide_size(B, over)
    mask = {"macroblock": synth.macroblock_mask(H, W, 3, 0.2), "few_lost": synth.iid_mask(H, W, 4, 1 / 256),
            "half_lost": synth.iid_mask(H, W, 5, 0.5), "all_known": np.ones((H, W), np.uint8)}[kind]
    t = torch.rand(H, W, device="cuda", generator=torch.Generator("cuda").manual_seed(B)) * 255
    m = torch.from_numpy(mask).cuda()
    kw = dict(block=B, border=(32 - B) // 2, iters=5)
    n = -(-H // B) * -(-W // B)
    seq = torch.zeros(n * 5, dtype=torch.int16, device="cuda")
    full = handle.reconstruct(t, m, seq_out=seq, **kw)
    got = handle.reconstruct(t, m, out=torch.full_like(t, -9.0), **kw)
    assert torch.equal(got, full)
    assert torch.equal(got[m != 0], t[m != 0])


def _inputs(H, W, seed, missing=0.55):
    g = torch.Generator("cuda").manual_seed(seed)
    t = torch.rand(H, W, device="cuda", generator=g) * 255
    return t, (torch.rand(H, W, device="cuda", generator=g) >= missing).to(torch.uint8)


@pytest.mark.parametrize("B", [2, 4, 8, 16])
def test_tile_copies_equal_plain_loads(handle, B):
    """Aligned rows (tile copies), rows whose pitch is not a multiple of 16 and
    dense rows (plain loads), with garbage beyond the width: bit for bit."""
    from paper_2202_13926_gb300 import fsr
    H, W = wide_size(B)
    t, m = _inputs(H, W, 3 * B)
    n = -(-H // B) * -(-W // B)
    res = []
    for P in (-(-W // 16) * 16 + 16, W + 1 if (W + 1) % 16 else W + 2, W):
        bi = torch.full((H, P), float("nan"), device="cuda")
        bm = torch.full((H, P), 1, dtype=torch.uint8, device="cuda")
        bo = torch.full((H, P), -5.0, device="cuda")
        bi[:, :W], bm[:, :W] = t, m
        seq = torch.full((n * 12,), -7, dtype=torch.int16, device="cuda")
        for s in (seq, None):   # with the indices every block is iterated; without, blocks may be copied
            fsr.fsr_reconstruct(handle.ptr, bi[:, :W], bm[:, :W],
                                fsr.make_params(block=B, border=(32 - B) // 2, iters=12, seq_out=s), bo[:, :W])
            handle.check_status()
            res.append((bo[:, :W].clone(), seq))
        assert torch.all(bo[:, W:] == -5.0)
    for out, seq in res[1:]:
        assert torch.equal(out, res[0][0])
        assert torch.equal(seq, res[0][1])
    assert torch.equal(res[0][0][m != 0], t[m != 0])


def test_many_calls_in_flight_on_two_streams(handle):
    """150 single-image calls on two streams, each with a table slot of its
    handle (there are 64), give the results of the calls made alone."""
    from paper_2202_13926_gb300 import fsr
    H, W = wide_size(4)
    ims = [_inputs(H, W, 40 + i) for i in range(5)]
    alone = [handle.reconstruct(t, m, iters=3) for t, m in ims]
    outs = [torch.full_like(ims[0][0], -1.0) for _ in range(150)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    p = fsr.make_params(iters=3)
    torch.cuda.synchronize()
    for j, out in enumerate(outs):
        fsr.fsr_reconstruct(handle.ptr, *ims[j % 5], p, out, streams[j % 2])
    torch.cuda.synchronize()
    for j, out in enumerate(outs):
        assert torch.equal(out, alone[j % 5]), j


def test_empty_blocks_are_counted_like_the_oracle(handle):
    import oracle
    import parity as PA
    from paper_2202_13926_gb300 import fsr
    H, W = wide_size(4)
    img = synth.sinusoid_image(H, W, seed=41)
    mask = synth.macroblock_mask(H, W, seed=42, lost=0.6, mb=40)
    n_ref = oracle.fsr_image_blocks(img, mask, K=2, rho=PA.RHO)["n_empty"]
    assert n_ref > 0
    t, m = torch.from_numpy(img).cuda(), torch.from_numpy(mask).cuda()
    fsr.fsr_empty_blocks(handle.ptr)   # reset
    handle.reconstruct(t, m, iters=2)
    assert fsr.fsr_empty_blocks(handle.ptr) == n_ref
    fsr.fsr_reconstruct_batch(handle.ptr, [fsr.image_desc(t, m, torch.empty_like(t), 2)], fsr.make_params(iters=2))
    assert fsr.fsr_empty_blocks(handle.ptr) == n_ref
