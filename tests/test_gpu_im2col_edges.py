"""Parity of im2col at the edges of its blocks: one column, fewer and more
columns than a block has threads, rows that step over several image rows and
images at once, a last run that is not full, runs of several passes, and
strides that leave rows and columns of the image unread."""
import numpy as np
import pytest

import oracle as O
import synth
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, host


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()


# (batch, channels, height, width, f, pad, stride)
CASES = [(300, 1, 1, 1, 1, 0, 1), (7, 1, 3, 5, 1, 0, 1), (5, 29, 2, 3, 3, 1, 1), (2, 257, 3, 1, 1, 0, 1),
         (3, 3, 9, 7, 5, 4, 3), (1, 1, 40, 40, 17, 16, 1), (11, 2, 4, 4, 4, 3, 5), (1000, 1, 33, 31, 2, 1, 1)]


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("cfg", CASES, ids=str)
def test_im2col_block_edges(ring, cfg):
    B, C, H, W, f, pad, stride = cfg
    x = synth.uniform(B + C + H, 1, 0, (B, C, H, W), ring.bits)
    Ho, Wo = (H - f + 2 * pad) // stride + 1, (W - f + 2 * pad) // stride + 1
    out = empty_like_ring((B * Ho * Wo, C * f * f), ring.words)
    abi.mpc_im2col(ring.k, ring.s, B, C, H, W, f, pad, stride, dev(x), out)
    assert np.array_equal(host(out), O.im2col(x, f, pad, stride, ring.bits))


@pytest.mark.gpu
def test_im2col_of_many_small_images_costs_what_its_bytes_do():
    """200,000 images of one value against one image of as many: the same bytes."""
    import torch

    def best(B, H, W):
        x = torch.zeros(B * H * W, dtype=torch.int64, device="cuda")
        out = torch.empty_like(x)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        t = []
        for _ in range(8):
            e[0].record()
            for _ in range(20):
                abi.mpc_im2col(32, 32, B, 1, H, W, 1, 0, 1, x, out)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        return min(t)
    assert best(200000, 1, 1) < 3 * best(1, 400, 500)
