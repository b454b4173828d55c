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
