"""Parity of the residue path of the ring GEMM (products modulo 16 or 31 small
moduli, rebuilt by the Chinese remainder theorem): equal to the oracle bit for
bit at the edges of its 256-row and 128- or 256-column tiles, its 64-deep
stages and 256-deep reductions, with odd sizes, with both operand orders, with
and without K splits, and for words that make every product largest."""
import numpy as np
import pytest

import oracle as O
import synth
from oracle import dealer
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, gpu_public_product, gpu_share, gpu_tag_full, host

CRT = 256      # the launch-table value of the path


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()
    yield
    abi.mpc_autotune_clear()


def _force(ring, M, K, N):
    L = abi.make_layer(M, K, N, ring.k, ring.s)
    abi.mpc_autotune_set(L, 1, tile_rows=CRT)
    assert abi.mpc_gemm_path(L) == 1 and abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3


SHAPES = [(synth.Z64, (256, 64, 256)), (synth.Z64, (257, 129, 255)), (synth.Z64, (9, 33, 17)),
          (synth.Z64, (300, 100, 130)), (synth.Z64, (20, 150, 600)), (synth.Z64, (255, 128, 128)),
          (synth.Z64, (40, 1500, 48)), (synth.Z128, (256, 32, 256)), (synth.Z128, (129, 70, 101)),
          (synth.Z128, (50, 97, 300)), (synth.Z128, (30, 500, 40))]


@pytest.mark.gpu
@pytest.mark.parametrize("ring,shape", SHAPES, ids=lambda x: str(x) if isinstance(x, tuple) else None)
def test_residue_path_parity(ring, shape):
    M, K, N = shape
    _force(ring, M, K, N)
    d = dealer.deal(ring, M, K, N, n=2, seed=M * 5 + K + N)
    for i, p in enumerate(d.parties):
        Z = gpu_share(ring, i, d.E, d.F, p.A, p.B, p.C)
        assert np.array_equal(Z, O.linear_share(ring.bits, i, d.E, d.F, p.A, p.B, p.C)), f"share party {i}"
        mZ = gpu_tag_full(ring, i, p.alpha, d.E, d.F, p.mA, p.mB, p.mC)
        assert np.array_equal(mZ, O.linear_tag_full(ring.bits, p.alpha, d.E, d.F, p.mA, p.mB, p.mC)), f"tag {i}"
    assert np.array_equal(gpu_public_product(ring, d.E, d.F), O.public_product(ring.bits, d.E, d.F))
    assert abi.mpc_device_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("top", [0x8000000000000000, 0x7FFFFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF, 0x77FFFFFFFFFFFFFF],
                         ids=hex)
def test_residue_path_extremes(ring, top):
    """Every word the same and the largest inner dimension, so that the integer
    product is as large as it gets (2K 2^126 or 2K 2^254): Z = 2K x^2 everywhere."""
    M, K, N = 640, 16384, 640
    L = abi.make_layer(M, K, N, ring.k, ring.s, 1, 2)
    abi.mpc_autotune_set(L, 1, tile_rows=CRT)
    low = 0xFFFFFFFFFFFFFFFF if top & 1 else 0
    x = top if ring.words == 1 else (top << 64) | low

    def mk(r, c, v):
        a = np.zeros((r, c) + ((2,) if ring.words == 2 else ()), dtype=np.uint64)
        if ring.words == 2:
            a[..., 0], a[..., 1] = v & (2**64 - 1), v >> 64
        else:
            a[...] = v
        return a
    E, F = dev(mk(M, K, x)), dev(mk(K, N, x))
    Z = empty_like_ring((M, N), ring.words)
    abi.mpc_linear_share(L, E, F, E, F, dev(mk(M, N, 0)), Z)
    assert np.array_equal(host(Z), mk(M, N, 2 * K * x * x % (1 << ring.bits)))
    assert abi.mpc_device_status() == 0


@pytest.mark.gpu
def test_residue_path_in_groups_and_small_workspaces():
    """A grouped call that mixes the paths equals the one-layer calls; a
    workspace that only covers the digit tiles is still accepted."""
    ring = synth.Z128
    abi.mpc_autotune_clear()
    shapes = [(512, 512, 512), (100, 64, 48), (4, 300, 64), (400, 640, 512), (2048, 72, 32)]
    Ls = [abi.make_layer(*s, ring.k, ring.s, 0, 2) for s in shapes]
    # two layers on the residue path, one on the tall digit tile, two on the integer pipes
    assert abi.mpc_launch_count_grouped(Ls, abi.MPC_WS_SHARE) == 2 * 3 + 2 + 2
    data, ptrs, want = [], [], []
    for L, (M, K, N) in zip(Ls, shapes):
        u = lambda tid, *s: dev(synth.uniform(M + N, tid, 0, s, 128))     # noqa: E731
        x = dict(E=u(1, M, K), F=u(2, K, N), A_i=u(3, M, K), B_i=u(4, K, N), C_i=u(5, M, N))
        data.append(x)
        w = empty_like_ring((M, N), 2)
        abi.mpc_linear_share(L, x["E"], x["F"], x["A_i"], x["B_i"], x["C_i"], w)
        want.append(host(w))
        ptrs.append(dict(x, Z_i=empty_like_ring((M, N), 2)))
    abi.mpc_linear_share_grouped(Ls, ptrs)
    for p, w in zip(ptrs, want):
        assert np.array_equal(host(p["Z_i"]), w)
    # the digit planes of the 512 x 512 x 512 layer: 32 bytes per element of [E | X]
    import torch
    ws = torch.empty(32 * 512 * 1024, dtype=torch.uint8, device="cuda")
    x, Z = data[0], empty_like_ring((512, 512), 2)
    abi.mpc_linear_share(Ls[0], x["E"], x["F"], x["A_i"], x["B_i"], x["C_i"], Z, ws=ws)
    assert np.array_equal(host(Z), want[0])
    assert abi.mpc_device_status() == 0


def test_residue_path_rule():
    """Where the built-in rule takes the path: large in both output dimensions
    (from about 600 in Z_2^64, 256 in Z_2^128), or odd N in Z_2^64."""
    abi.mpc_autotune_clear()

    def crt(M, K, N, bits=64):
        L = abi.make_layer(M, K, N, bits // 2, bits // 2)
        n = abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3
        assert not n or abi.mpc_gemm_path(L) == 1
        return n
    assert crt(2048, 1024, 4096) and crt(4096, 4096, 4096) and crt(1000, 999, 1001)
    assert crt(512, 512, 512, 128) and crt(1024, 2304, 256, 128)
    assert not crt(128, 4096, 4096) and not crt(32768, 576, 64) and not crt(1024, 576, 64)
    assert not crt(8, 4096, 4096, 128) and not crt(32768, 576, 64, 128) and not crt(64, 128, 64)
    assert not crt(1024, 16385, 1024), "2K beyond the proven range"


def test_residue_path_rule_in_groups():
    """A group's layers take the path by its own estimate in both rings, also where
    the digit tiles could run them."""
    abi.mpc_autotune_clear()

    def crt(M, K, N, bits):
        Ls = [abi.make_layer(M, K, N, bits // 2, bits // 2)]
        n = abi.mpc_launch_count_grouped(Ls * 2, abi.MPC_WS_SHARE)
        assert n in (6, 2)      # three launches per layer, or a launch pair for both
        return n == 6
    assert crt(1129, 1692, 1468, 64) and crt(2048, 1024, 4096, 64) and crt(1000, 999, 1001, 64)
    assert crt(1024, 2304, 256, 128) and crt(512, 512, 512, 128)
    assert not crt(1024, 576, 64, 64) and not crt(128, 4096, 4096, 64) and not crt(512, 512, 512, 64)
    # 1.9 GB of planes: a launch pair of its own on the digit tiles, and no planes in the workspace
    big = abi.make_layer(2048, 4096, 4096)
    assert abi.mpc_launch_count(big, abi.MPC_WS_SHARE) == 3
    assert abi.mpc_launch_count_grouped([big], abi.MPC_WS_SHARE) == 2
    size = abi.mpc_workspace_size_grouped([big], abi.MPC_WS_SHARE)
    assert size == abi.mpc_workspace_size_grouped([big], abi.MPC_WS_SHARE | abi.MPC_WS_LEAST)
    abi.mpc_autotune_set(big, 1, tile_rows=CRT)
    assert abi.mpc_launch_count_grouped([big], abi.MPC_WS_SHARE) == 3
    assert abi.mpc_workspace_size_grouped([big], abi.MPC_WS_SHARE) > size
    abi.mpc_autotune_clear()
