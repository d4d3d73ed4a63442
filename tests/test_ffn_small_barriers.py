"""The cluster barriers of the f32 feed-forward block on a few tokens are aligned ones: a warp has to reach them whole.  Where a product has too few terms or too
many outputs to share a sum between threads, it ends in a loop that a warp's lanes leave at different turns."""
import os
import re

import pytest

from test_gpu_einsum import layout, mtf  # noqa: F401

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_02084_b200", "csrc", "ffn_f32_small.cu")


def test_every_aligned_barrier_comes_right_behind_the_warp_barrier():
    text = open(SOURCE).read()
    at = [m.start() for m in re.finditer(r'asm volatile\("barrier\.cluster\.\w+\.\w+\.aligned', text)]
    assert len(at) >= 2 and all(text[:i].rstrip().endswith("__syncwarp();") for i in at)


# hidden units a block, outputs of y: 8 and 9 in one part, 13 and 36, 17 and 300: the last warp has 9, 4 and 12 lanes at work
@pytest.mark.gpu
@pytest.mark.parametrize("T,D,F,E", [(9, 16, 64, 6), (33, 64, 104, 8), (40, 8, 136, 60)])
def test_partly_filled_warps_before_the_barriers(mtf, T, D, F, E):  # noqa: F811
    import torch
    from test_gpu_ffn_small import block, check, run
    lay = layout(mtf, [("all", 1)], [])
    t = block(T, D, F, E)
    assert run(mtf, lay, t) == 2
    check(t)
    for _ in range(20):
        again = block(T, D, F, E)
        assert run(mtf, lay, again) == 2
        assert all(torch.equal(t[k], again[k]) for k in t)
