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
