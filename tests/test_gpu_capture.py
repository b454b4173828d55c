"""Calls of the integer pipes and of the residue path under stream capture: what
they record, and that a replay with new operands in the same buffers gives the
oracle's bits."""
import ctypes

import numpy as np
import pytest

import oracle as O
import synth
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()
    abi.mpc_autotune_clear()
    yield
    abi.mpc_autotune_clear()


def nodes(call):
    """Graph nodes that call(stream) records."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    st, graph, n = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(st.cuda_stream), 2) == 0      # relaxed
    try:
        call(st)
    finally:
        end = cu.cuStreamEndCapture(ctypes.c_void_p(st.cuda_stream), ctypes.byref(graph))
    assert end == 0 and cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert cu.cuGraphDestroy(graph) == 0
    return n.value


def operands(ring, M, K, N, seed):
    u = lambda t, *s: synth.uniform(seed, t, 1, s, ring.bits)     # noqa: E731
    return u(1, M, K), u(2, K, N), u(3, M, K), u(4, K, N), u(5, M, N)


@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("shape", [(64, 128, 64), (4, 512, 100)], ids=str)
def test_split_target_of_the_launch_table(ring, shape):
    """The built-in rule adds the K splits of small layers up in a cluster: one
    kernel.  An entry with a split target gets splits that meet in Z: a copy of C
    and the kernel."""
    M, K, N = shape
    L = abi.make_layer(M, K, N, ring.k, ring.s)
    x = operands(ring, M, K, N, M + K)
    d, Z = [dev(t) for t in x], empty_like_ring((M, N), ring.words)
    for waves, want in ((0, 1), (1, 2), (4, 2)):
        abi.mpc_autotune_set(L, 0, 0, waves)
        abi.mpc_linear_share(L, *d, Z)
        assert np.array_equal(host(Z), O.linear_share(ring.bits, 0, *x)), waves
        assert nodes(lambda st: abi.mpc_linear_share(L, *d, Z, stream=st)) == want
    abi.mpc_autotune_clear()


@pytest.mark.parametrize("ring,shapes", [
    (synth.Z64, [(700, 300, 701)]), (synth.Z128, [(400, 640, 512)]), (synth.Z64, [(64, 128, 64)]),
    (synth.Z128, [(512, 512, 512), (100, 64, 48), (4, 300, 64), (400, 640, 512), (2048, 72, 32)])],
    ids=["residues_z64", "residues_z128", "cluster_z64", "group_z128"])
def test_replay(ring, shapes):
    import torch
    Ls = [abi.make_layer(*s, ring.k, ring.s) for s in shapes]
    bufs = [[dev(t) for t in operands(ring, *s, 1)] + [empty_like_ring(s[::2], ring.words)] for s in shapes]
    names = ("E", "F", "A_i", "B_i", "C_i", "Z_i")
    ws = torch.empty(max(abi.mpc_workspace_size_grouped(Ls, abi.MPC_WS_SHARE), 256), dtype=torch.uint8, device="cuda")

    def call():
        if len(Ls) == 1:
            abi.mpc_linear_share(Ls[0], *bufs[0], ws=ws)
        else:
            abi.mpc_linear_share_grouped(Ls, [dict(zip(names, b)) for b in bufs], ws=ws)
    call()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    for seed in (2, 3):
        x = [operands(ring, *s, seed) for s in shapes]
        for b, t in zip(bufs, x):
            for dst, src in zip(b, t):
                dst.copy_(dev(src))
            b[-1].zero_()
        g.replay()
        for b, t, s in zip(bufs, x, shapes):
            assert np.array_equal(host(b[-1]), O.linear_share(ring.bits, 0, *t)), (seed, s)
    assert abi.mpc_device_status() == 0
