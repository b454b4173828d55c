"""CompactTag passes that take several rows per warp (layers with many rows or
narrow outputs) and the check of many rows: equal to the oracle bit for bit at
the edges of the four-row groups, with odd sizes and either side empty."""
import numpy as np
import pytest

import oracle as O
import synth
from paper_2311_04406_gb300 import abi, build

from gpuhelp import dev, empty_like_ring, gpu_check_compact, gpu_tag_compact, host

pytestmark = pytest.mark.gpu

# 9728 rows: the passes switch to four rows per warp
SHAPES = [(9727, 64, 64), (9728, 64, 64), (9729, 65, 33), (9730, 130, 256), (9731, 129, 257), (9733, 63, 7),
          (9800, 0, 5), (40000, 27, 10), (5, 9740, 66), (9, 9730, 1), (4863, 4865, 34)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()


def _inputs(ring, M, K, N, seed):
    t = synth.TID
    u = lambda n, *s: synth.uniform(seed, t[n], 0, s, ring.bits)     # noqa: E731
    return dict(alpha=u("alpha", 1).reshape((1,) if ring.words == 1 else (1, 2)), E=u("E", M, K), F=u("F", K, N),
                mA=u("mA", M, K), mB=u("mB", K, N), mC=u("mC", M, N), mR=u("mR", M, N), Dt=u("Dt", M, N),
                chi=u("chi", N), chi_hat=u("chi_hat", M))


@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_many_rows(ring, shape):
    M, K, N = shape
    x = _inputs(ring, M, K, N, seed=M + 3 * K + N)
    mZ, mDc, Dc = gpu_tag_compact(ring, 1, x["alpha"], x["E"], x["F"], x["mA"], x["mB"], x["mC"], x["mR"], x["Dt"],
                                  x["chi"])
    rmDc, rDc, _ = O.compact_tag(ring.bits, x["alpha"], x["E"], x["F"], x["mA"], x["mB"], x["mC"], x["mR"], x["Dt"],
                                 x["chi"])
    assert np.array_equal(mZ, O.optmac(ring.bits, x["alpha"], x["mR"], x["Dt"]))
    assert np.array_equal(Dc, rDc) and np.array_equal(mDc, rmDc)
    cs = gpu_check_compact(ring, x["alpha"], x["chi_hat"], Dc, mDc)
    assert np.array_equal(cs.reshape(-1), O.check_compact(ring.bits, x["alpha"], x["chi_hat"], rDc, rmDc).reshape(-1))


@pytest.mark.parametrize("ring", [synth.Z64, synth.Z128], ids=["z64", "z128"])
def test_many_rows_grouped(ring):
    """One grouped call over all the shapes equals the one-layer calls, the truncated tag included."""
    shapes = [s for s in SHAPES if s[1] > 0]
    Ls = [abi.make_layer(*s, ring.k, ring.s) for s in shapes]
    for mode in (abi.MPC_TAG_COMPACT, abi.MPC_TAG_COMPACT_TRUNC):
        ptrs, want = [], []
        for L, (M, K, N) in zip(Ls, shapes):
            x = {k: dev(v) for k, v in _inputs(ring, M, K, N, seed=M + K).items()}
            d = dict(alpha_i=x["alpha"], E=x["E"], F=x["F"], mA_i=x["mA"], mB_i=x["mB"], mC_i=x["mC"], mR_i=x["mR"],
                     Dtilde=x["Dt"], chi=x["chi"])
            mk = lambda: dict(mZ_i=empty_like_ring((M, N), ring.words) if mode == abi.MPC_TAG_COMPACT else None,
                              mDc_i=empty_like_ring((M,), ring.words), Dc=empty_like_ring((M,), ring.words))   # noqa: E731
            o, p = mk(), mk()
            abi.mpc_linear_tag(L, mode, **d, **o)
            want.append(o)
            ptrs.append(dict(d, **p))
        abi.mpc_linear_tag_grouped(Ls, mode, ptrs)
        for o, p in zip(want, ptrs):
            for n, t in o.items():
                assert t is None or np.array_equal(host(t), host(p[n])), n
