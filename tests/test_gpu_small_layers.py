"""Parity of the integer-pipe kernels around their choices: K splits that fit
one cluster and ones that need atomics, splits without rows, up to 16 columns
and more, odd and even widths, every row count of the GEMV, short and long K
of wide layers, with a public coefficient, a tag's key, and no addend."""
import numpy as np
import pytest

import oracle as O
import synth
from oracle import dealer
from paper_2311_04406_gb300 import abi, build

from gpuhelp import gpu_public_product, gpu_share, gpu_tag_full


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()
    yield
    abi.mpc_autotune_clear()


SHAPES = [(1, 1, 1), (9, 8, 16), (9, 9, 17), (16, 33, 64), (33, 70, 40), (17, 128, 65), (40, 400, 16), (130, 129, 9),
          (16, 3000, 10), (64, 128, 64), (200, 184, 168), (1, 64, 64), (1, 65, 71), (2, 600, 300), (3, 129, 257),
          (4, 535, 76), (5, 1023, 256), (7, 181, 1322), (8, 299, 368), (8, 1100, 1200), (6, 5000, 31), (1, 20000, 10)]


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_integer_pipe_parity(ring, shape):
    M, K, N = shape
    abi.mpc_autotune_set(abi.make_layer(M, K, N, ring.k, ring.s), 0, 8, 0)
    d = dealer.deal(ring, M, K, N, n=2, seed=M + 7 * K + N)
    for i, p in enumerate(d.parties):
        Z = gpu_share(ring, i, d.E, d.F, p.A, p.B, p.C)
        assert np.array_equal(Z, O.linear_share(ring.bits, i, d.E, d.F, p.A, p.B, p.C)), f"share party {i}"
    p = d.parties[0]
    mZ = gpu_tag_full(ring, 0, p.alpha, d.E, d.F, p.mA, p.mB, p.mC)
    assert np.array_equal(mZ, O.linear_tag_full(ring.bits, p.alpha, d.E, d.F, p.mA, p.mB, p.mC))
    assert np.array_equal(gpu_public_product(ring, d.E, d.F), O.public_product(ring.bits, d.E, d.F))
