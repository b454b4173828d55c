"""The native marshalling (csrc/binding.c) takes what the general path takes and
refuses what it refuses; without it the general path runs every call."""
import pytest

from paper_2311_04406_gb300 import abi, build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()


def test_calls_run_without_the_native_marshalling(monkeypatch, tmp_path):
    import torch
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_binding.so"))
    monkeypatch.setattr(abi, "_lib", None)
    monkeypatch.setattr(abi, "_nat", None)
    assert abi.load() is not None and abi._nat is None
    t = torch.zeros(8, dtype=torch.int64)
    with pytest.raises(ValueError, match="dst"):
        abi.mpc_transpose(32, 32, 2, 8, torch.zeros(16, dtype=torch.int64), t)
    with pytest.raises(ValueError, match=r"ins\[0\]"):
        abi.mpc_lincomb(32, 32, [1], [t[:4]], t)


def test_build_without_python_headers(monkeypatch, tmp_path):
    so = tmp_path / "_binding.so"
    so.write_bytes(b"of an older build")
    monkeypatch.setattr(build, "BINDING", str(so))
    monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    assert build.binding_headers() is None
    build.build_binding(build.binding_headers())
    assert not so.exists()
    assert build.build() == build.LIB and not so.exists()


class _Buf:
    """Stands in for a tensor; on_read runs when its size is asked for."""

    def __init__(self, nbytes, on_read=None, contiguous=True, address=0x1000):
        self._n, self._on, self._c, self._a = nbytes, on_read, contiguous, address

    @property
    def nbytes(self):
        if self._on:
            self._on()
        return self._n

    def is_contiguous(self):
        return self._c

    def data_ptr(self):
        return self._a

    def numel(self):
        return self._n // 8


def _calls(M, K, N, words):
    """name -> (arguments before the operands, operands with their bytes, arguments after) of the
    single calls, workspace and stream included."""
    e = 8 * words
    L = abi.make_layer(M, K, N, 32 * words, 32 * words)
    mk, kn, mn = M * K * e, K * N * e, M * N * e
    ws = (0x100000, 1 << 30)
    k = 32 * words
    return {
        "share": ((L,), [mk, kn, mk, kn, mn, mn], ws + (0,)),
        "share_trunc": ((L,), [mk, kn, mk, kn, mn, mn], ws + (0,)),
        "tag": ((L, abi.MPC_TAG_COMPACT), [e, mk, kn, mk, kn, mn, mn, mn, N * e, mn, M * e, M * e], ws + (0,)),
        "check": ((L, abi.MPC_CHECK_BATCHREC), [e, mn, mn, mn, e], ws + (0,)),
        "public_product": ((L,), [mk, kn, mn], ws + (0,)),
        "optmac_trunc": ((L, 5), [e, mn, mn, mn, mn, mn, mn], (0,)),
        "batchrec_mask": ((k, k, M, N), [mn] * 8, (0,)),
        "transpose": ((k, k, M, N), [mn, mn], (0,)),
        "im2col": ((k, k, M, 1, 3, 3, 3, 1, 1), [M * 9 * e, M * 9 * 9 * e], (0,)),
    }


@pytest.mark.hidden_gpu
@pytest.mark.parametrize("words", [1, 2])
def test_operands_are_checked(words):
    """Full operands reach the library (which fails: no GPU); one byte short, not
    contiguous or not an integer leaves the call to the general path."""
    for name, (pre, sizes, post) in _calls(16, 24, 32, words).items():
        f = getattr(abi._nat, name)
        ok = [_Buf(n) for n in sizes]
        assert f(*pre, *ok, *post) == abi.MPC_E_CUDA, name
        assert f(*pre, *[0x1000] * len(ok), *post) == abi.MPC_E_CUDA, name
        assert f(*pre, None, *ok[1:], *post) == abi.MPC_E_NULL, name       # a missing operand is the library's to refuse
        for i, n in enumerate(sizes):
            for bad in (_Buf(n - 1), _Buf(n, contiguous=False)):
                assert f(*pre, *ok[:i], bad, *ok[i + 1:], *post) is None, (name, i)
        for i in range(len(pre)):
            if isinstance(pre[i], int):
                assert f(*pre[:i], float(pre[i]), *pre[i + 1:], *ok, *post) is None, (name, i)
        assert f(*pre, *ok, *post) == abi.MPC_E_CUDA, name


@pytest.mark.hidden_gpu
def test_grouped_operands_are_checked():
    M, K, N = 16, 24, 32
    L = abi.make_layer(M, K, N)
    nat, ws = abi._nat, (0x100000, 1 << 30)
    sizes = dict(alpha_i=1, E=M * K, F=K * N, mA_i=M * K, mB_i=K * N, mC_i=M * N, mR_i=M * N, Dtilde=M * N, chi=N,
                 mZ_i=M * N, mDc_i=M, Dc=M)
    calls = {
        "share": (abi._share_elems(M, K, N), lambda Ls, ps: nat.share_grouped(Ls, ps, *ws, 0)),
        "tag": (sizes, lambda Ls, ps: nat.tag_grouped(Ls, abi.MPC_TAG_COMPACT, ps, *ws, 0)),
        "check": (dict(alpha_i=1, chi_hat=M, Dc=M, mDc_i=M, cs_i=1), lambda Ls, ps: nat.check_grouped(Ls, ps, 0)),
    }
    for name, (elems, call) in calls.items():
        full = lambda: {k: _Buf(8 * n) for k, n in elems.items()}      # noqa: E731
        assert call([L, L], [full(), full()]) == abi.MPC_E_CUDA, name
        assert call((L, L), [full(), full()]) is None and call([L, L], (full(), full())) is None, name
        assert call([L, L], [full()]) is None and call([], []) is None, name
        for k, n in elems.items():
            for bad in (_Buf(8 * n - 1), _Buf(8 * n, contiguous=False)):
                assert call([L, L], [full(), dict(full(), **{k: bad})]) is None, (name, k)
            assert call([L, L], [full(), dict(full(), **{k: None})]) == abi.MPC_E_NULL, (name, k)
    assert nat.tag_grouped([L], 1.0, [{k: _Buf(8 * n) for k, n in sizes.items()}], *ws, 0) is None


@pytest.mark.hidden_gpu
def test_lists_that_change_while_they_are_read():
    nat = abi._nat
    ins = []
    ins[:] = [_Buf(64, on_read=ins.clear), _Buf(64)]
    assert nat.lincomb(32, 32, [1, 1], ins, _Buf(64), 0) is None
    row = []
    row[:] = [_Buf(64, on_read=row.clear), _Buf(64)]
    assert nat.lincomb_grouped(32, 32, [1, 1], [row, [_Buf(64)] * 2], [_Buf(64)] * 2, None, 0) is None
    outs = []
    outs[:] = [_Buf(64, on_read=outs.clear), _Buf(64)]
    assert nat.lincomb_grouped(32, 32, [1], [[_Buf(64)]] * 2, outs, None, 0) is None
    L = abi.make_layer(2, 2, 2)
    e = abi._share_elems(2, 2, 2)
    ptrs = []
    ptrs[:] = [{k: _Buf(8 * n, on_read=ptrs.clear) for k, n in e.items()}, {k: _Buf(8 * n) for k, n in e.items()}]
    assert nat.share_grouped([L, L], ptrs, 0x100000, 1 << 30, 0) is None
    p = {}
    p.update({k: _Buf(8 * n, on_read=p.clear) for k, n in e.items()})
    assert nat.share_grouped([L], [p], 0x100000, 1 << 30, 0) == abi.MPC_E_NULL      # the operands are gone


@pytest.mark.gpu
def test_refusals_on_the_gpu():
    """The same through the public calls: the general path raises, nothing is launched."""
    import torch
    assert abi._nat is not None
    M, K, N = 16, 24, 32
    L = abi.make_layer(M, K, N)
    t = lambda *s: torch.ones(s, dtype=torch.int64, device="cuda")      # noqa: E731
    ops = dict(E=t(M, K), F=t(K, N), A_i=t(M, K), B_i=t(K, N), C_i=t(M, N), Z_i=t(M, N) * 7)
    for k in ops:
        short = dict(ops, **{k: ops[k].flatten()[:-1]})
        with pytest.raises(ValueError, match=k):
            abi.mpc_linear_share(L, *short.values())
        with pytest.raises(ValueError, match=k):
            abi.mpc_linear_share_grouped([L, L], [ops, short])
        missing = dict(ops, **{k: None})
        with pytest.raises(abi.MpcError, match="NULL"):
            abi.mpc_linear_share(L, *missing.values())
        with pytest.raises(abi.MpcError, match="NULL"):
            abi.mpc_linear_share_grouped([L], [missing])
    with pytest.raises(ValueError, match="contiguous"):
        abi.mpc_linear_share(L, *dict(ops, F=t(N, K).t()).values())
    assert bool((ops["Z_i"] == 7).all())
    abi.mpc_linear_share_grouped((L,), (ops,))         # tuples: the general path
    assert bool((ops["Z_i"] == 1 + 3 * K).all())       # C + E.B + A.F + E.F of ones, party 0
    al, P, Zf, mZf = t(1), t(M, N), t(M, N), t(M, N)
    abi.mpc_optmac_trunc(L, 4.0, al, P, P, P, P, Zf, mZf)      # converted as ever
    want = [Zf.clone(), mZf.clone()]
    abi.mpc_optmac_trunc(L, 4, al, P, P, P, P, Zf, mZf)
    assert torch.equal(want[0], Zf) and torch.equal(want[1], mZf)
