"""The check sum of an opening around the sizes where a thread's elements come
four at a time, and one at a time for the rest."""
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


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("n", [1, 511, 1537, 2048, 2049, 4095, 4097, 6143, 12293])
def test_batchrec_check_sum(ring, n):
    u = lambda t, shape: synth.uniform(n, t, 0, shape, ring.bits)
    alpha, chi, W, mW = u(1, (1,)), u(2, (n, 1)), u(3, (n, 1)), u(4, (n, 1))
    L = abi.make_layer(n, 1, 1, ring.k, ring.s)
    cs = empty_like_ring((1,), ring.words)
    abi.mpc_tag_check(L, abi.MPC_CHECK_BATCHREC, dev(alpha), dev(chi), dev(W), dev(mW), cs)
    assert np.array_equal(host(cs).reshape(-1), np.asarray(O.check_batchrec(ring.bits, alpha, chi, W, mW)).reshape(-1))


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("rows", [(1,), (2048,), (2049,), (4095, 1, 2050), (16385, 40), (700, 33000, 5)], ids=str)
def test_compact_check_rows(ring, rows):
    """One block up to 2048 rows, a cluster of them beyond; grouped checks mix both."""
    layers, ptrs, want = [], [], []
    for j, M in enumerate(rows):
        u = lambda t, shape: synth.uniform(M + j, t, 0, shape, ring.bits)
        alpha, chi, Dc, mDc = u(1, (1,)), u(2, (M,)), u(3, (M,)), u(4, (M,))
        layers.append(abi.make_layer(M, 1, 1, ring.k, ring.s))
        want.append(np.asarray(O.check_compact(ring.bits, alpha, chi, Dc, mDc)).reshape(-1))
        ptrs.append(dict(alpha_i=dev(alpha), chi_hat=dev(chi), Dc=dev(Dc), mDc_i=dev(mDc),
                         cs_i=empty_like_ring((1,), ring.words)))
        cs = empty_like_ring((1,), ring.words)
        abi.mpc_tag_check(layers[-1], abi.MPC_CHECK_COMPACT, ptrs[-1]["alpha_i"], ptrs[-1]["chi_hat"], ptrs[-1]["Dc"],
                          ptrs[-1]["mDc_i"], cs)
        assert np.array_equal(host(cs).reshape(-1), want[-1])
    abi.mpc_tag_check_grouped(layers, ptrs)
    for q, w in zip(ptrs, want):
        assert np.array_equal(host(q["cs_i"]).reshape(-1), w)
