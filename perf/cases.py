"""Performance cases: one party's online work for SPDZ2k linear layers.

Each case is one call pattern of a program that uses the library, on seeded
inputs that are resident on the GPU, through the public binding
(paper_2311_04406_gb300.abi).  Shares, triple shares, tags and opened matrices
are uniform ring words, which is exactly the distribution of real protocol
data; keys and combiners are uniform in [0, 2^s).  Every output is an integer.

Kinds of case:
  layer     one layer: the share, then its tag (CompactTag with its check, or
            the full SPDZ2k tag); "share": False leaves the tag path alone
  conv      a convolution: im2col of the opened image, the mask share and the
            mask's tag share, then the layer as above
  trunc     a truncated layer: share, public product, OptMAC&Trunc, the
            truncated compact tag and its check
  backward  training: transposes of the reused masks, then the two gradient
            layers (grad X = G W^T, grad W = X^T G), each with CompactTag
  grouped   every linear layer of a network (or a batch of unrelated layers)
            in grouped calls: shares, openings, CompactTag tags, checks
  opening   Pi_BatchRec of a matrix: masking for two parties, the opening, and
            the seeded tag check
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_04406_gb300 import abi

RINGS = {64: (32, 32), 128: (64, 64)}     # ring width -> (k, s)
GROUPED_OUT = ("Z", "Dt", "mZ", "mDc", "Dc", "cs")


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the smallest call: a 64-row dense layer with 128 inputs and 64 outputs; latency and launches
        dict(name="dense_64x128x64", kind="layer", ring=64, M=64, K=128, N=64, party=0, share=True, tag="compact"),
        # one 3x3 convolution of a CIFAR-sized network at batch 1 (im2col 1024 x 576 x 64)
        dict(name="conv3x3_64c_32x32", kind="conv", ring=64, batch=1, channels=64, height=32, width=32, out=64, f=3,
             pad=1, stride=1, party=1, tag="compact"),
        # a 4096 x 4096 dense layer at batch 128 under the full SPDZ2k tag (the baseline protocol)
        dict(name="dense_128x4096x4096_full", kind="layer", ring=64, M=128, K=4096, N=4096, party=0, share=True,
             tag="full"),
        # the CompactTag tag and check of the same layer by themselves: the pass over memory
        dict(name="dense_128x4096x4096_tag", kind="layer", ring=64, M=128, K=4096, N=4096, party=1, share=False,
             tag="compact"),
        # a Transformer encoder's FFN up-projection (H = 1024, 2048 rows) with truncation
        dict(name="ffn_up_2048x1024x4096_trunc", kind="trunc", ring=64, M=2048, K=1024, N=4096, party=0, f=16),
        # the backward pass of the 4096 x 4096 dense layer at batch 128
        dict(name="dense_128x4096x4096_backward", kind="backward", ring=64, M=128, K=4096, N=4096, party=1),
        # VGG16 inference on 32x32 images: one image (latency) and a batch of 32 (throughput)
        dict(name="vgg16_b1", kind="grouped", ring=64, net="vgg16", batch=1, party=0),
        dict(name="vgg16_b32", kind="grouped", ring=64, net="vgg16", batch=32, party=1),
        # ResNet-18 inference in Z_2^128, the serving ring: one image and a batch of 16
        dict(name="resnet18_b1_z128", kind="grouped", ring=128, net="resnet18", batch=1, party=1),
        dict(name="resnet18_b16_z128", kind="grouped", ring=128, net="resnet18", batch=16, party=0),
        # unrelated layers of uneven, mostly ragged shapes in one grouped call, as a batching server collects them
        dict(name="uneven_48", kind="grouped", ring=64, net="uneven", batch=48, pick=7, party=0),
        # the opening and check of a 2047 x 1025 matrix in Z_2^128 (both sizes odd)
        dict(name="opening_2047x1025_z128", kind="opening", ring=128, M=2047, N=1025),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "conv", "trunc", "backward", "grouped", "grouped", "opening"])
    ring = rng.choice([64, 128])
    party = rng.randrange(2)
    if kind == "conv":
        f = rng.choice([1, 3, 5])
        return dict(kind=kind, ring=ring, batch=_log_int(rng, 1, 32), channels=_log_int(rng, 3, 128),
                    height=rng.randint(8, 36), width=rng.randint(8, 36), out=_log_int(rng, 16, 256), f=f,
                    pad=f // 2, stride=rng.choice([1, 1, 2]), party=party, tag="compact")
    if kind == "opening":
        return dict(kind=kind, ring=ring, M=_log_int(rng, 16, 4096), N=_log_int(rng, 16, 2048))
    if kind == "grouped":
        net = rng.choice(["vgg16", "resnet18", "uneven"])
        if net == "uneven":
            return dict(kind=kind, ring=64, net=net, batch=_log_int(rng, 8, 48), pick=rng.randrange(1 << 20),
                        party=party)
        return dict(kind=kind, ring=ring, net=net, batch=_log_int(rng, 1, 16 if ring == 64 else 8), party=party)
    lo, hi = {"layer": (1, 4096), "trunc": (32, 2048), "backward": (8, 512)}[kind]
    while True:
        M, K, N = _log_int(rng, lo, hi), _log_int(rng, 32, 4096), _log_int(rng, 32, 4096)
        if M * K * N <= (1 << 31):
            break
    case = dict(kind=kind, ring=ring, M=M, K=K, N=N, party=party)
    if kind == "layer":
        case.update(share=True, tag=rng.choice(["compact", "compact", "full"]))
    if kind == "trunc":
        case["f"] = rng.choice([12, 16, 20])
    return case


# ---------------------------------------------------------------------------
# layer shapes

def _conv_rows(h, w, f, pad, stride):
    return ((h - f + 2 * pad) // stride + 1) * ((w - f + 2 * pad) // stride + 1)


def _vgg16(batch):
    plan = [64, 64, 0, 128, 128, 0, 256, 256, 256, 0, 512, 512, 512, 0, 512, 512, 512]
    out, side, cin = [], 32, 3
    for c in plan:
        if c == 0:
            side //= 2
            continue
        out.append((side * side * batch, cin * 9, c))
        cin = c
    return out + [(batch, 512, 4096), (batch, 4096, 4096), (batch, 4096, 10)]


def _resnet18(batch):
    out, side, cin = [(1024 * batch, 27, 64)], 32, 64
    for stage, c in enumerate([64, 128, 256, 512]):
        for blk in range(2):
            if stage > 0 and blk == 0:
                side //= 2
                out.append((side * side * batch, cin, c))      # the 1x1 downsample
            out += [(side * side * batch, cin * 9, c), (side * side * batch, c * 9, c)]
            cin = c
    return out + [(batch, 512, 10)]


def _uneven(count, pick):
    """`count` layers, M log-uniform in [1, 4096], K and N log-uniform in
    [64, 2048], two thirds of them moved off the multiples of 8."""
    r = np.random.default_rng(pick)
    out = []
    for i in range(count):
        m = int(round(math.exp(r.uniform(0.0, math.log(4096.0)))))
        k, n = (int(round(math.exp(r.uniform(math.log(64.0), math.log(2048.0))))) for _ in range(2))
        if i % 3 == 0:
            k, n = -(-k // 8) * 8, -(-n // 8) * 8
        elif i % 3 == 1:
            n += n & 1
        out.append((max(1, m), k, n))
    return out


def _layers(case):
    kind = case["kind"]
    if kind == "grouped":
        return {"vgg16": _vgg16, "resnet18": _resnet18}[case["net"]](case["batch"]) if case["net"] != "uneven" \
            else _uneven(case["batch"], case["pick"])
    if kind == "conv":
        rows = case["batch"] * _conv_rows(case["height"], case["width"], case["f"], case["pad"], case["stride"])
        return [(rows, case["channels"] * case["f"] ** 2, case["out"])]
    if kind == "backward":
        M, K, N = case["M"], case["K"], case["N"]
        return [(M, N, K), (K, M, N)]
    return [(case["M"], case["K"], case["N"])]


# ---------------------------------------------------------------------------
# inputs

class _Words:
    """Uniform ring words on the GPU from a seed, one call after another."""

    def __init__(self, seed, ring):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
        self.w, self.s = ring // 64, ring // 2

    def ring(self, *shape):
        return torch.randint(-2**63, 2**63 - 1, shape + ((2,) if self.w == 2 else ()), dtype=torch.int64,
                             device="cuda", generator=self.g)

    def key(self, n):
        """n ring elements uniform in [0, 2^s)"""
        if self.w == 1:
            return torch.randint(0, 2**32, (n,), dtype=torch.int64, device="cuda", generator=self.g)
        out = self.ring(n)
        out[:, 1] = 0
        return out

    def out(self, *shape):
        return torch.zeros(shape + ((2,) if self.w == 2 else ()), dtype=torch.int64, device="cuda")

    def packed(self, counts):
        """one output buffer and its per-layer parts, each on a 16-byte boundary"""
        off = np.concatenate([[0], np.cumsum([_even(n) for n in counts])])
        flat = self.out(int(off[-1]))
        return flat, [flat[int(a):int(a) + n] for a, n in zip(off, counts)]


def _even(n):
    return n + (n & 1)


def _compact_inputs(r, M, K, N):
    """operands of the tag path beyond E and F"""
    return dict(mB=r.ring(K, N), mC=r.ring(M, N), mR=r.ring(M, N), Dt=r.ring(M, N), chi=r.key(N), chi_hat=r.key(M))


def _inputs(case, seed):
    r = _Words(seed, case["ring"])
    kind = case["kind"]
    if kind == "opening":
        M, N = case["M"], case["N"]
        d = {f"{n}{i}": r.ring(M, N) for i in range(2) for n in ("X", "A", "R", "mX", "mA", "mR")}
        d["alpha"] = r.key(1)
        d["seed"] = torch.randint(-2**63, 2**63 - 1, (1,), dtype=torch.int64, device="cuda", generator=r.g)
        return d, r
    d = dict(alpha=r.key(1))
    if kind == "conv":
        (M, K, N), = _layers(case)
        img = (case["batch"], case["channels"], case["height"], case["width"])
        d.update(E_img=r.ring(*img), A_img=r.ring(*img), mA_img=r.ring(*img), F=r.ring(K, N), B=r.ring(K, N),
                 C=r.ring(M, N))
        d.update(_compact_inputs(r, M, K, N))
    elif kind == "backward":
        M, K, N = case["M"], case["K"], case["N"]
        # E = X - A, F = W - B of the forward pass; G = grad Z is masked by A2: E2 = G - A2
        d.update(E=r.ring(M, K), A=r.ring(M, K), mA=r.ring(M, K), F=r.ring(K, N), B=r.ring(K, N), mB=r.ring(K, N),
                 E2=r.ring(M, N), A2=r.ring(M, N), mA2=r.ring(M, N))
        for j, (m, k, n) in enumerate(_layers(case)):
            d.update({f"C_{j}": r.ring(m, n), f"mC_{j}": r.ring(m, n), f"mR_{j}": r.ring(m, n),
                      f"Dt_{j}": r.ring(m, n), f"chi_{j}": r.key(n), f"chi_hat_{j}": r.key(m)})
    elif kind == "grouped":
        d["layers"] = []
        for (M, K, N) in _layers(case):
            q = dict(E=r.ring(M, K), F=r.ring(K, N), A=r.ring(M, K), B=r.ring(K, N), C=r.ring(M, N), mA=r.ring(M, K),
                     R=r.ring(M, N), Z_other=r.ring(M, N), R_other=r.ring(M, N))
            q.update(mB=r.ring(K, N), mC=r.ring(M, N), mR=r.ring(M, N), chi=r.key(N), chi_hat=r.key(M))
            d["layers"].append(q)
    else:
        (M, K, N), = _layers(case)
        d.update(E=r.ring(M, K), F=r.ring(K, N), mA=r.ring(M, K))
        if kind == "trunc" or case["share"]:
            d.update(A=r.ring(M, K), B=r.ring(K, N), C=r.ring(M, N))
        if kind == "layer" and case["tag"] == "full":
            d.update(mB=r.ring(K, N), mC=r.ring(M, N))
        else:
            d.update(_compact_inputs(r, M, K, N))
        if kind == "trunc":
            d.update(Rf=r.ring(M, N), mRf=r.ring(M, N))
    return d, r


def prepare(case, seed):
    d, r = _inputs(case, seed)
    k, s = RINGS[case["ring"]]
    st = dict(case=case, d=d, k=k, s=s)
    if case["kind"] == "opening":
        M, N = case["M"], case["N"]
        st["L"] = [abi.make_layer(M, 1, N, k, s, 0, 2)]
        st["o"] = {n: r.out(M, N) for n in ("W0", "W1", "mW0", "mW1", "V")}
        st["o"]["cs"] = r.out(1)
        need = abi.mpc_workspace_size(st["L"][0], abi.MPC_WS_CHECK_BATCHREC)
    else:
        shapes = _layers(case)
        st["L"] = [abi.make_layer(M, K, N, k, s, case["party"], 2) for (M, K, N) in shapes]
        if case["kind"] == "grouped":      # a program keeps one buffer per kind of output
            sizes = dict(Z=[M * N for (M, K, N) in shapes], mDc=[M for (M, K, N) in shapes], cs=[1] * len(shapes))
            sizes.update(mZ=sizes["Z"], Dt=sizes["Z"], Dc=sizes["mDc"])
            st["flat"], parts = {}, {}
            for n in GROUPED_OUT:
                st["flat"][n], parts[n] = r.packed(sizes[n])
            st["o"] = [{n: parts[n][i] for n in GROUPED_OUT} for i in range(len(shapes))]
        else:
            st["o"] = [dict(Z=r.out(M, N), mZ=r.out(M, N), mDc=r.out(M), Dc=r.out(M), cs=r.out(1),
                            **({"P": r.out(M, N), "Zf": r.out(M, N)} if case["kind"] == "trunc" else {}))
                       for (M, K, N) in shapes]
        if case["kind"] == "conv":
            (M, K, N), = shapes
            st["t"] = {n: r.out(M, K) for n in ("E", "A", "mA")}
        if case["kind"] == "backward":
            M, K, N = case["M"], case["K"], case["N"]
            st["t"] = {n: r.out(N, K) for n in ("FT", "BT", "mBT")}
            st["t"].update({n: r.out(K, M) for n in ("ET", "AT", "mAT")})
        if case["kind"] == "grouped":
            need = max(abi.mpc_workspace_size_grouped(st["L"], w)
                       for w in (abi.MPC_WS_SHARE, abi.MPC_WS_TAG_COMPACT))
        else:
            need = max(abi.mpc_workspace_size(L, w) for L in st["L"]
                       for w in (abi.MPC_WS_SHARE, abi.MPC_WS_TAG_FULL, abi.MPC_WS_TAG_COMPACT,
                                 abi.MPC_WS_PUBLIC_PRODUCT, abi.MPC_WS_SHARE_TRUNC))
    st["ws"] = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
    return st


# ---------------------------------------------------------------------------
# one pass

def _compact(L, o, d, alpha, ws, mode=abi.MPC_TAG_COMPACT):
    """CompactTag tag and check of one layer (operands by name in d)"""
    mz = o["mZ"] if mode == abi.MPC_TAG_COMPACT else None
    abi.mpc_linear_tag(L, mode, alpha, d["E"], d["F"], d["mA"], d["mB"], d["mC"], mz, mR_i=d["mR"], Dtilde=d["Dt"],
                       chi=d["chi"], mDc_i=o["mDc"], Dc=o["Dc"], ws=ws)
    abi.mpc_tag_check(L, abi.MPC_CHECK_COMPACT, alpha, d["chi_hat"], o["Dc"], o["mDc"], o["cs"])


def run(st):
    case, d, o, ws, k, s = st["case"], st["d"], st["o"], st["ws"], st["k"], st["s"]
    kind = case["kind"]
    if kind == "opening":
        L, M, N = st["L"][0], case["M"], case["N"]
        for i in range(2):
            abi.mpc_batchrec_mask(k, s, M, N, d[f"X{i}"], d[f"A{i}"], d[f"R{i}"], d[f"mX{i}"], d[f"mA{i}"],
                                  d[f"mR{i}"], o[f"W{i}"], o[f"mW{i}"])
        abi.mpc_lincomb(k, s, [1, 1], [o["W0"], o["W1"]], o["V"])
        abi.mpc_tag_check(L, abi.MPC_CHECK_BATCHREC_SEEDED, d["alpha"], d["seed"], o["V"], o["mW0"], o["cs"], ws=ws)
        return o
    if kind == "grouped":
        Ls, q = st["L"], d["layers"]
        abi.mpc_linear_share_grouped(Ls, [dict(E=x["E"], F=x["F"], A_i=x["A"], B_i=x["B"], C_i=x["C"], Z_i=y["Z"])
                                          for x, y in zip(q, o)], ws=ws)
        # D~ = (R_0 - Z_0) + (R_1 - Z_1), the other party's matrices as received
        abi.mpc_lincomb_grouped(k, s, [1, -1, 1, -1], [[x["R"], y["Z"], x["R_other"], x["Z_other"]]
                                                       for x, y in zip(q, o)], [y["Dt"] for y in o])
        abi.mpc_linear_tag_grouped(Ls, abi.MPC_TAG_COMPACT,
                                   [dict(alpha_i=d["alpha"], E=x["E"], F=x["F"], mA_i=x["mA"], mB_i=x["mB"],
                                         mC_i=x["mC"], mR_i=x["mR"], Dtilde=y["Dt"], chi=x["chi"], mZ_i=y["mZ"],
                                         mDc_i=y["mDc"], Dc=y["Dc"]) for x, y in zip(q, o)], ws=ws)
        abi.mpc_tag_check_grouped(Ls, [dict(alpha_i=d["alpha"], chi_hat=x["chi_hat"], Dc=y["Dc"], mDc_i=y["mDc"],
                                            cs_i=y["cs"]) for x, y in zip(q, o)])
        return st["flat"]
    if kind == "backward":
        t, M, K, N = st["t"], case["M"], case["K"], case["N"]
        for src, dst, r, c in (("F", "FT", K, N), ("B", "BT", K, N), ("mB", "mBT", K, N),
                               ("E", "ET", M, K), ("A", "AT", M, K), ("mA", "mAT", M, K)):
            abi.mpc_transpose(k, s, r, c, d[src], t[dst])
        # grad X: left G (E2, A2), right W^T; grad W: left X^T, right G
        sides = [dict(E=d["E2"], A=d["A2"], mA=d["mA2"], F=t["FT"], B=t["BT"], mB=t["mBT"]),
                 dict(E=t["ET"], A=t["AT"], mA=t["mAT"], F=d["E2"], B=d["A2"], mB=d["mA2"])]
        for j, (L, x, y) in enumerate(zip(st["L"], sides, o)):
            abi.mpc_linear_share(L, x["E"], x["F"], x["A"], x["B"], d[f"C_{j}"], y["Z"], ws=ws)
            x.update({n: d[f"{n}_{j}"] for n in ("mC", "mR", "Dt", "chi", "chi_hat")})
            _compact(L, y, x, d["alpha"], ws)
        return o
    L, y = st["L"][0], o[0]
    if kind == "trunc":
        abi.mpc_linear_share_trunc(L, d["E"], d["F"], d["A"], d["B"], d["C"], y["Z"], ws=ws)
        abi.mpc_public_product(L, d["E"], d["F"], y["P"], ws=ws)
        abi.mpc_optmac_trunc(L, case["f"], d["alpha"], d["Rf"], d["mRf"], d["Dt"], y["P"], y["Zf"], y["mZ"])
        _compact(L, y, d, d["alpha"], ws, abi.MPC_TAG_COMPACT_TRUNC)
        return o
    x = d
    if kind == "conv":
        x = dict(d, **st["t"])
        for n in ("E", "A", "mA"):
            abi.mpc_im2col(k, s, case["batch"], case["channels"], case["height"], case["width"], case["f"],
                           case["pad"], case["stride"], d[n + "_img"], st["t"][n])
    if kind == "conv" or case["share"]:
        abi.mpc_linear_share(L, x["E"], x["F"], x["A"], x["B"], x["C"], y["Z"], ws=ws)
    if case["tag"] == "full":
        abi.mpc_linear_tag(L, abi.MPC_TAG_FULL, x["alpha"], x["E"], x["F"], x["mA"], x["mB"], x["mC"], y["mZ"], ws=ws)
    else:
        _compact(L, y, x, x["alpha"], ws)
    return o


# ---------------------------------------------------------------------------
# the least work of one pass

def work(case):
    """bytes: every input once and every output once; flops: two per ring
    multiply-add (2 M K N ring products per share or full tag)."""
    e, kind = case["ring"] // 8, case["kind"]
    if kind == "opening":
        n = case["M"] * case["N"]
        return {"bytes": e * 17 * n, "flops": 20 * n}
    b = f = 0
    for (M, K, N) in _layers(case):
        mk, kn, mn = M * K, K * N, M * N
        compact = 2 * (4 * mn + 2 * kn + 2 * mk)
        if kind == "trunc":
            b += e * (3 * mk + 3 * kn + 10 * mn)
            f += 2 * 3 * mk * N + compact
        elif kind == "grouped":
            b += e * (3 * mk + 3 * kn + 9 * mn)
            f += 2 * 2 * mk * N + compact
        elif kind == "layer" and case["tag"] == "full":
            b += e * (3 * mk + 3 * kn + 4 * mn)
            f += 2 * 4 * mk * N
        elif kind == "layer" and not case["share"]:
            b += e * (2 * mk + 2 * kn + 4 * mn)
            f += compact
        else:
            b += e * (3 * mk + 3 * kn + 6 * mn)
            f += 2 * 2 * mk * N + compact
    if kind == "backward":      # the shared operands are inputs once; the transposes are written once
        M, K, N = case["M"], case["K"], case["N"]
        b += e * 3 * (K * N + M * K)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same values from plain 64-bit host arithmetic

def _mul(a, b):
    """elementwise ring product; a, b: (lo, hi) of uint64 (hi None in Z_2^64)"""
    with np.errstate(over="ignore"):
        lo = a[0] * b[0]
        if a[1] is None:
            return lo, None
        m = np.uint64(0xFFFFFFFF)
        t = np.uint64(32)
        al, ah, bl, bh = a[0] & m, a[0] >> t, b[0] & m, b[0] >> t
        mid = ah * bl + ((al * bl) >> t)
        mid2 = al * bh + (mid & m)
        hi = ah * bh + (mid >> t) + (mid2 >> t) + a[0] * b[1] + a[1] * b[0]
        return lo, hi


def _add(a, b):
    with np.errstate(over="ignore"):
        lo = a[0] + b[0]
        return (lo, None) if a[1] is None else (lo, a[1] + b[1] + (lo < a[0]).astype(np.uint64))


def _neg(a):
    with np.errstate(over="ignore"):
        lo = ~a[0] + np.uint64(1)
        return (lo, None) if a[1] is None else (lo, ~a[1] + (lo == 0).astype(np.uint64))


def _sub(a, b):
    return _add(a, _neg(b))


def _limbs(a):
    """16-bit limbs as float64 matrices"""
    out = []
    for w in a:
        if w is not None:
            out += [torch.from_numpy(((w >> np.uint64(16 * j)) & np.uint64(0xFFFF)).astype(np.float64))
                    for j in range(4)]
    return out


def _dot(a, b):
    """ring matrix product: 16-bit limb products in float64 (exact below 2^53),
    recombined in wrapping 64-bit words"""
    la, lb = _limbs(a), _limbs(b)
    n = len(la)
    shape = (a[0].shape[0], b[0].shape[1])
    acc = (np.zeros(shape, np.uint64), None if a[1] is None else np.zeros(shape, np.uint64))
    for t in range(n):
        p = sum(la[i] @ lb[t - i] for i in range(t + 1)).numpy().astype(np.uint64)     # below 2^53
        sh = 16 * t
        lo = p << np.uint64(sh) if sh < 64 else np.zeros_like(p)
        if a[1] is None:
            acc = _add(acc, (lo, None))
        else:
            hi = p << np.uint64(sh - 64) if sh >= 64 else (p >> np.uint64(64 - sh) if sh > 0 else np.zeros_like(p))
            acc = _add(acc, (lo, hi))
    return acc


def _host(t, ring):
    a = t.cpu().numpy().view(np.uint64)
    return (a, None) if ring == 64 else (np.ascontiguousarray(a[..., 0]), np.ascontiguousarray(a[..., 1]))


def _dev(a):
    """back to the binding's layout"""
    x = a[0] if a[1] is None else np.stack([a[0], a[1]], axis=-1)
    return torch.from_numpy(np.ascontiguousarray(x).view(np.int64))


def _at(a, f):
    return f(a[0]), None if a[1] is None else f(a[1])


def _vec(m, v):
    return _at(_dot(m, _at(v, lambda x: x.reshape(-1, 1))), lambda x: x.reshape(-1))


def _zero(ring, *shape):
    return np.zeros(shape, np.uint64), None if ring == 64 else np.zeros(shape, np.uint64)


def _full(E, F, X, B, C, c):
    """C + E.B + X.F + c E.F (c a one-element ring value or None)"""
    z = _add(_add(C, _dot(E, B)), _dot(X, F))
    return z if c is None else _add(z, _mul(_dot(E, F), c))


def _exact_compact(ring, x, alpha, out, trunc=False):
    """the CompactTag tag and check of one layer"""
    if not trunc:
        out["mZ"] = _sub(x["mR"], _mul(x["Dt"], alpha))
    mb, fc = _vec(x["mB"], x["chi"]), _vec(x["F"], x["chi"])
    zc = _add(_add(_vec(x["mC"], x["chi"]), _vec(x["E"], mb)), _vec(x["mA"], fc))
    if not trunc:
        zc = _add(zc, _mul(_vec(x["E"], fc), alpha))
    out["mDc"] = _sub(_vec(x["mR"], x["chi"]), zc)
    out["Dc"] = _vec(x["Dt"], x["chi"])
    v = _mul(x["chi_hat"], _sub(_mul(out["Dc"], alpha), out["mDc"]))
    out["cs"] = _sum(v)
    return out


def _sum(v):
    """wrapping sum of a vector, as one element"""
    one = np.ones((1, v[0].size), np.uint64), None if v[1] is None else np.zeros((1, v[0].size), np.uint64)
    return _at(_dot(one, _at(v, lambda x: x.reshape(-1, 1))), lambda x: x.reshape(-1))


def _im2col(a, f, pad, stride):
    def one(x):
        x = np.pad(x, ((0, 0), (0, 0), (pad, pad), (pad, pad)))
        v = np.lib.stride_tricks.sliding_window_view(x, (f, f), axis=(2, 3))[:, :, ::stride, ::stride]
        b, c, oy, ox = v.shape[:4]
        return np.ascontiguousarray(v.transpose(0, 2, 3, 1, 4, 5)).reshape(b * oy * ox, c * f * f)
    return _at(a, one)


def exact(case, seed):
    ring, kind = case["ring"], case["kind"]
    prods = {64: 10, 128: 36}[ring]
    if kind != "opening":
        per = {"trunc": 3, "grouped": 3}.get(kind, 4)
        if per * prods * sum(M * K * N for (M, K, N) in _layers(case)) > 1.2e11:
            return None                    # over some seconds of host matrix products
    d, _ = _inputs(case, seed)
    h = lambda t: _host(t, ring)           # noqa: E731
    zeros = lambda *n: _zero(ring, *n)     # noqa: E731
    if kind == "opening":
        o = {}
        for i in range(2):
            o[f"W{i}"] = _add(_sub(h(d[f"X{i}"]), h(d[f"A{i}"])), h(d[f"R{i}"]))
            o[f"mW{i}"] = _add(_sub(h(d[f"mX{i}"]), h(d[f"mA{i}"])), h(d[f"mR{i}"]))
        o["V"] = _add(o["W0"], o["W1"])
        n = case["M"] * case["N"]
        with np.errstate(over="ignore"):
            z = np.uint64(d["seed"].cpu().numpy().view(np.uint64)[0]) + \
                np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z ^= z >> np.uint64(31)
        chi = (z & np.uint64(0xFFFFFFFF), None) if ring == 64 else (z, np.zeros_like(z))
        flat = lambda a: _at(a, lambda x: x.reshape(-1))     # noqa: E731
        o["cs"] = _sum(_mul(chi, _sub(flat(o["mW0"]), _mul(flat(o["V"]), h(d["alpha"])))))
        order = ("W0", "W1", "mW0", "mW1", "V", "cs")
        return {n_: _dev(o[n_]) for n_ in order}
    alpha = h(d["alpha"])
    one = (np.ones(1, np.uint64), None if ring == 64 else np.zeros(1, np.uint64))
    share_c = one if case["party"] == 0 else None
    outs = []
    shapes = _layers(case)

    def blank(M, N):
        return dict(Z=zeros(M, N), mZ=zeros(M, N), mDc=zeros(M), Dc=zeros(M), cs=zeros(1))

    if kind == "grouped":
        for (M, K, N), q in zip(shapes, d["layers"]):
            x = {n: h(t) for n, t in q.items()}
            y = blank(M, N)
            y["Z"] = _full(x["E"], x["F"], x["A"], x["B"], x["C"], share_c)
            y["Dt"] = x["Dt"] = _add(_sub(x["R"], y["Z"]), _sub(x["R_other"], x["Z_other"]))
            outs.append(_exact_compact(ring, x, alpha, y))
        pad = lambda w: np.concatenate([w.reshape(-1), np.zeros(w.size & 1, np.uint64)])     # noqa: E731
        return {n: torch.cat([_dev(_at(y[n], pad)) for y in outs]) for n in GROUPED_OUT}
    elif kind == "backward":
        v = {n: h(t) for n, t in d.items()}
        T = lambda a: _at(a, lambda x: np.ascontiguousarray(x.T))     # noqa: E731
        sides = [dict(E=v["E2"], A=v["A2"], mA=v["mA2"], F=T(v["F"]), B=T(v["B"]), mB=T(v["mB"])),
                 dict(E=T(v["E"]), A=T(v["A"]), mA=T(v["mA"]), F=v["E2"], B=v["A2"], mB=v["mA2"])]
        for j, ((M, K, N), x) in enumerate(zip(shapes, sides)):
            y = blank(M, N)
            y["Z"] = _full(x["E"], x["F"], x["A"], x["B"], v[f"C_{j}"], share_c)
            x.update({n: v[f"{n}_{j}"] for n in ("mC", "mR", "Dt", "chi", "chi_hat")})
            outs.append(_exact_compact(ring, x, alpha, y))
    else:
        (M, K, N), = shapes
        x = {n: h(t) for n, t in d.items()}
        y = blank(M, N)
        if kind == "conv":
            for n in ("E", "A", "mA"):
                x[n] = _im2col(x[n + "_img"], case["f"], case["pad"], case["stride"])
        if kind == "trunc":
            y["Z"] = _full(x["E"], x["F"], x["A"], x["B"], x["C"], None)
            y["P"] = _dot(x["E"], x["F"])
            k, f = RINGS[ring][0], case["f"]
            # the k-bit value floor-divided by 2^f (k = 32: low half of the word; k = 64: the low word)
            low = lambda a: ((a[0] & np.uint64(0xFFFFFFFF)) if k == 32 else a[0]) >> np.uint64(f)     # noqa: E731
            wide = lambda w: (w, None if ring == 64 else np.zeros_like(w))     # noqa: E731
            tau = _sub(wide(low(y["P"])), wide(low(x["Dt"])))
            y["Zf"] = _add(x["Rf"], tau) if case["party"] == 0 else x["Rf"]
            y["mZ"] = _add(x["mRf"], _mul(tau, alpha))
            _exact_compact(ring, x, alpha, y, trunc=True)
        else:
            if kind == "conv" or case["share"]:
                y["Z"] = _full(x["E"], x["F"], x["A"], x["B"], x["C"], share_c)
            if case["tag"] == "full":
                y["mZ"] = _full(x["E"], x["F"], x["mA"], x["mB"], x["mC"], alpha)
            else:
                _exact_compact(ring, x, alpha, y)
        outs.append(y)
    return [{n: _dev(a) for n, a in y.items()} for y in outs]
