"""Parity of the tile epilogue of the row digit kernel, which moves the tile's
rows by bulk copies: tiles computed whole (with and without an addend, one
after another in a CTA), pieces of split tiles, ragged last rows and columns,
both tile heights, and layers of one grouped launch."""
import numpy as np
import pytest

import oracle as O
import synth
from oracle import dealer
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, gpu_public_product, gpu_share, host


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()
    yield
    abi.mpc_autotune_clear()


# whole tiles (more tiles than SMs, one interval each), then split ones
SHAPES = [(synth.Z64, (1281, 40, 1022)), (synth.Z64, (640, 9, 2050)), (synth.Z64, (130, 1000, 70)),
          (synth.Z64, (40, 700, 34)), (synth.Z128, (901, 30, 333)), (synth.Z128, (1290, 5, 497)),
          (synth.Z128, (129, 300, 49)), (synth.Z128, (65, 401, 17))]


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [64, 128])
@pytest.mark.parametrize("ring,shape", SHAPES, ids=lambda x: str(x) if isinstance(x, tuple) else None)
def test_row_tile_epilogue(ring, shape, rows):
    M, K, N = shape
    L = abi.make_layer(M, K, N, ring.k, ring.s)
    abi.mpc_autotune_set(L, 1, tile_rows=rows)
    d = dealer.deal(ring, M, K, N, n=2, seed=M + 3 * K + N)
    p = d.parties[1]
    want = O.linear_share(ring.bits, 1, d.E, d.F, p.A, p.B, p.C)
    assert np.array_equal(gpu_share(ring, 1, d.E, d.F, p.A, p.B, p.C), want)
    assert np.array_equal(gpu_public_product(ring, d.E, d.F), O.public_product(ring.bits, d.E, d.F))
    assert abi.mpc_device_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
def test_row_tile_epilogue_grouped(ring):
    """Layers of different heights and widths share one launch."""
    shapes = [(1025, 20, 260), (128, 600, 34), (514, 33, 130)]
    layers, ptrs, want = [], [], []
    for j, (M, K, N) in enumerate(shapes):
        L = abi.make_layer(M, K, N, ring.k, ring.s)
        abi.mpc_autotune_set(L, 1, tile_rows=128)
        layers.append(abi.make_layer(M, K, N, ring.k, ring.s, 1, 2))
        d = dealer.deal(ring, M, K, N, n=2, seed=71 + j)
        p = d.parties[1]
        Z = empty_like_ring((M, N), ring.words)
        ptrs.append(dict(E=dev(d.E), F=dev(d.F), A_i=dev(p.A), B_i=dev(p.B), C_i=dev(p.C), Z_i=Z))
        want.append(O.linear_share(ring.bits, 1, d.E, d.F, p.A, p.B, p.C))
    abi.mpc_linear_share_grouped(layers, ptrs)
    for q, w in zip(ptrs, want):
        assert np.array_equal(host(q["Z_i"]), w)
    assert abi.mpc_device_status() == 0
