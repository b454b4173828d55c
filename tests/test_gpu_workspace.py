"""What the layers of the residue path ask of the caller's workspace: the built-in
rule takes the path only where the workspace serves it, and a call that ran
without it (integer pipes: odd N in Z_2^64) still runs in any workspace."""
import ctypes

import numpy as np
import pytest

import synth
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, host

ODD = (700, 300, 701)      # Z_2^64 with odd N, residue path by the built-in rule


@pytest.fixture(scope="module")
def lib():
    build.build()
    abi.mpc_autotune_clear()
    yield abi.load()
    abi.mpc_autotune_clear()


@pytest.mark.hidden_gpu
def test_workspace_is_judged_by_the_path_that_runs(lib):
    L = abi.make_layer(*ODD)
    need = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE)
    assert abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3 and need > 0
    p = [0x1000] * 6
    share = lambda ws: lib.mpc_linear_share(ctypes.byref(L), *p, ws, need, None)   # noqa: E731
    # gets past validation (and fails at the launch: no GPU here)
    assert share(0x10010) == abi.MPC_E_CUDA
    assert share(None) == abi.MPC_E_CUDA
    # an entry that demands the path is held to its workspace
    abi.mpc_autotune_set(L, 1, tile_rows=256)
    assert share(0x10010) == abi.MPC_E_ALIGN
    assert share(None) == abi.MPC_E_WORKSPACE
    abi.mpc_autotune_clear()


@pytest.mark.gpu
def test_unaligned_workspace_gives_the_same_result(lib):
    import torch
    M, K, N = ODD
    L = abi.make_layer(M, K, N)
    u = lambda tid, *s: dev(synth.uniform(M + N, tid, 0, s, 64))     # noqa: E731
    x = (u(1, M, K), u(2, K, N), u(3, M, K), u(4, K, N), u(5, M, N))
    buf = torch.empty(abi.mpc_workspace_size(L, abi.MPC_WS_SHARE) + 256, dtype=torch.uint8, device="cuda")
    out = []
    for ws in (buf, buf[16:]):
        Z = empty_like_ring((M, N), 1)
        abi.mpc_linear_share(L, *x, Z, ws=ws)
        out.append(host(Z))
    assert np.array_equal(out[0], out[1])
    assert abi.mpc_device_status() == 0
