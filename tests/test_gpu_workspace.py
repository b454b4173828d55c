"""What the layers of the residue path ask of the caller's workspace: they take the
path only where the workspace serves it, and a call that ran without it (integer
pipes: odd N in Z_2^64) still runs in any workspace."""
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
def test_workspace_is_held_to_the_path_that_runs(lib):
    L = abi.make_layer(*ODD)
    need = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE)
    assert abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3 and need > 0
    p = [0x1000] * 6
    share = lambda ws: lib.mpc_linear_share(ctypes.byref(L), *p, ws, need, None)   # noqa: E731
    # gets past validation (and fails at the launch: no GPU here)
    assert share(0x10010) == abi.MPC_E_CUDA
    assert share(None) == abi.MPC_E_CUDA
    # also when a table entry names the path
    abi.mpc_autotune_set(L, 1, tile_rows=256)
    assert share(0x10010) == abi.MPC_E_CUDA and share(None) == abi.MPC_E_CUDA
    # the digit tiles hold the workspace to their needs as ever
    L = abi.make_layer(64, 256, 256)
    digits = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE)
    abi.mpc_autotune_set(L, 1, tile_rows=256)
    assert abi.mpc_workspace_size(L, abi.MPC_WS_SHARE) > digits      # its planes, for callers that ask now
    need = digits
    assert share(0x10100) == abi.MPC_E_CUDA
    assert share(0x10010) == abi.MPC_E_ALIGN and share(None) == abi.MPC_E_WORKSPACE
    need -= 1
    assert share(0x10100) == abi.MPC_E_WORKSPACE
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


def test_grouped_workspace_sizes(lib):
    """The digit planes of all layers, or the residue planes of one: a group whose
    layers run as digits reserves no residue planes for them."""
    size = lambda shapes, bits: abi.mpc_workspace_size_grouped(      # noqa: E731
        [abi.make_layer(*s, bits // 2, bits // 2) for s in shapes], abi.MPC_WS_SHARE)
    for shape, bits in (((2048, 1024, 4096), 64), ((1129, 1692, 1468), 64), ((512, 512, 512), 128)):
        one = size([shape], bits)
        assert one == abi.mpc_workspace_size(abi.make_layer(*shape, bits // 2, bits // 2), abi.MPC_WS_SHARE)
        digits = size([shape] * 12, bits) - size([shape] * 11, bits)
        assert digits < one                      # the layer's own call may run as residues
        for n in (1, 2, 6, 11):
            assert size([shape] * n, bits) == max(one, n * digits)
    assert size([ODD] * 9, 64) == size([ODD], 64)     # no digit planes: one set of residue planes


@pytest.mark.gpu
@pytest.mark.parametrize("ring,shapes", [
    (synth.Z128, [(512, 512, 512), (100, 64, 48), (4, 300, 64), (400, 640, 512), (2048, 72, 32), (640, 512, 300)]),
    (synth.Z64, [ODD, (300, 200, 96), (900, 400, 901), (20, 300, 33), (1100, 64, 66)])], ids=["z128", "z64"])
def test_residue_layers_share_their_planes(lib, ring, shapes):
    """Residue layers of a group in the same planes, which overlay the digit planes,
    in every workspace from the smallest on: all on the path, some, none."""
    import torch
    Ls = [abi.make_layer(*s, ring.k, ring.s, 1, 2) for s in shapes]
    data, want = [], []
    for L, (M, K, N) in zip(Ls, shapes):
        u = lambda tid, *s: dev(synth.uniform(M + N, tid, 0, s, ring.bits))     # noqa: E731
        x = dict(E=u(1, M, K), F=u(2, K, N), A_i=u(3, M, K), B_i=u(4, K, N), C_i=u(5, M, N))
        data.append(x)
        w = empty_like_ring((M, N), ring.words)
        abi.mpc_linear_share(L, *x.values(), w)
        want.append(host(w))
    full = abi.mpc_workspace_size_grouped(Ls, abi.MPC_WS_SHARE)
    # digit planes: what a group of many copies grows by
    many = lambda n: abi.mpc_workspace_size_grouped(Ls * n, abi.MPC_WS_SHARE)      # noqa: E731
    digits = many(40) - many(39)
    crt = sorted(abi.mpc_workspace_size(L, abi.MPC_WS_SHARE) for L, s in zip(Ls, shapes)
                 if abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3)
    sizes = {full, max(digits, 256)} | {b for b in crt if b >= digits}
    assert len(crt) >= 2 and len(sizes) >= 2
    for nbytes in sorted(sizes):
        Zs = [empty_like_ring(s[::2], ring.words) for s in shapes]
        for rep in range(2):
            abi.mpc_linear_share_grouped(Ls, [dict(x, Z_i=Z) for x, Z in zip(data, Zs)],
                                         ws=torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
        for Z, w, s in zip(Zs, want, shapes):
            assert np.array_equal(host(Z), w), (nbytes, s)
    assert abi.mpc_device_status() == 0


def test_binding_falls_back_to_the_least_workspace(lib, monkeypatch):
    """A workspace allocated by the binding: the residue planes where they fit, what
    the other paths need where they do not; nothing is kept after the call."""
    import torch
    L = abi.make_layer(2048, 1024, 4096)
    full = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE)
    least = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE | abi.MPC_WS_LEAST)
    assert 0 < least < full // 4
    G = [L, abi.make_layer(*ODD)]
    assert abi.mpc_workspace_size_grouped(G, abi.MPC_WS_SHARE) == full
    assert abi.mpc_workspace_size_grouped(G, abi.MPC_WS_SHARE | abi.MPC_WS_LEAST) == least
    for which in (abi.MPC_WS_TAG_COMPACT, abi.MPC_WS_CHECK_BATCHREC):        # one size
        assert abi.mpc_workspace_size(L, which | abi.MPC_WS_LEAST) == abi.mpc_workspace_size(L, which)

    limit, asked = full, []
    abi._alloc_ws.__dict__.pop("keep", None)

    def empty(n, dtype=None, device=None):
        asked.append(n)
        if n > limit:
            raise torch.cuda.OutOfMemoryError("out of memory")
        return torch.zeros(1)
    monkeypatch.setattr(torch, "empty", empty)
    assert abi._ws(L, abi.MPC_WS_SHARE, None)[1] == full
    limit = full - 1
    assert abi._ws(L, abi.MPC_WS_SHARE, None)[1] == least
    assert abi._ws_grouped(G, abi.MPC_WS_SHARE, None)[1] == least
    assert asked == [full, full, least, full, least]
    limit = 0
    assert abi._ws(abi.make_layer(*ODD), abi.MPC_WS_SHARE, None) == (None, 0, None)     # integer pipes
    with pytest.raises(torch.cuda.OutOfMemoryError):
        abi._ws(L, abi.MPC_WS_SHARE, None)
    assert not hasattr(abi._alloc_ws, "keep")


@pytest.mark.gpu
def test_share_runs_where_only_the_digit_planes_fit(lib):
    import torch
    M, K, N = 2048, 1024, 4096
    L = abi.make_layer(M, K, N)
    u = lambda tid, *s: dev(synth.uniform(M + N, tid, 0, s, 64))     # noqa: E731
    x = (u(1, M, K), u(2, K, N), u(3, M, K), u(4, K, N), u(5, M, N))
    Z = [empty_like_ring((M, N), 1) for _ in range(2)]
    abi.mpc_linear_share(L, *x, Z[0])
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    room = abi.mpc_workspace_size(L, abi.MPC_WS_SHARE | abi.MPC_WS_LEAST) + (64 << 20)
    try:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + room) / total)
        abi.mpc_linear_share(L, *x, Z[1])
        torch.cuda.synchronize()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert np.array_equal(host(Z[0]), host(Z[1]))
    assert abi.mpc_device_status() == 0


@pytest.mark.gpu
def test_autotune_without_room_for_the_residue_planes(lib):
    """The residue candidate is left out, and the layer is tuned among the others."""
    import torch
    M, K, N = 2048, 1024, 4096
    L = abi.make_layer(M, K, N)
    assert abi.mpc_autotune([L]) == 1 and abi.mpc_autotune_choice(L)[4] == 256     # with room
    abi.mpc_autotune_clear()
    operands = 8 * (2 * M * K + 2 * K * N + 2 * M * N)
    room = operands + abi.mpc_workspace_size(L, abi.MPC_WS_SHARE | abi.MPC_WS_LEAST) + (256 << 20)
    assert room < operands + abi.mpc_workspace_size(L, abi.MPC_WS_SHARE)
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        assert abi.mpc_autotune([L]) == 1
    finally:
        del fill
        torch.cuda.empty_cache()
    assert abi.mpc_autotune_choice(L)[0] == 1 and abi.mpc_autotune_choice(L)[4] != 256
    abi.mpc_autotune_clear()


def test_what_the_queries_report(lib):
    """mpc_gemm_path and mpc_launch_count tell what runs in a full workspace,
    mpc_autotune_choice the table's entry or the rule's choice without the residue
    path."""
    for shape, bits, other in ((ODD, 64, (0, 0)), ((2048, 1024, 4096), 64, (1, 128)), ((512, 512, 512), 128, (1, 128))):
        L = abi.make_layer(*shape, bits // 2, bits // 2)
        assert abi.mpc_gemm_path(L) == 1 and abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3
        assert abi.mpc_autotune_choice(L)[::4] == other and not abi.mpc_autotune_choice(L)[3]
        abi.mpc_autotune_set(L, 1, 8, 0, tile_rows=256)
        assert abi.mpc_autotune_choice(L) == (1, 8, 0, True, 256) and abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 3
        if bits == 128:
            abi.mpc_autotune_set(L, 1, 8, 0, tile_rows=128)
            assert abi.mpc_autotune_choice(L)[4] == 128 and abi.mpc_launch_count(L, abi.MPC_WS_SHARE) == 2
        abi.mpc_autotune_clear()
