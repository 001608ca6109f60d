"""The work that programs have this library do, as a list of cases that can be timed.

Eight kinds of pass, each through the public calls of ``paper_2211_10482_b200``:

  moment2   the packed covariance X^T X of a table of samples, on request reconstructed to the symmetric
            matrix that a solver takes (linear regression, PCA)
  moment3   the packed third moment of a table
  moment4   the packed fourth moment of a table
  poly      the three blocks of a degree-2 polynomial-regression covariance of one batch, each added to
            the running sums of the batches before it, in packed form (covariance creation and addition)
  mttkrp    MTTKRP on a tensor stored for i <= j only
  ttm       TTM on a block-diagonal or an upper-triangular tensor
  chain     a dense operand packed, multiplied with a packed one (THP), added to a third, reconstructed
            once at the end of the chain
  copy      a dense array packed and unpacked again (encode and decode), every layout and element size

``mode`` is the precision that the caller asks for: "f32" (the default of every call), "tf32", "split",
"bf16".  Values are what standardised features and factor matrices look like: N(0,1), with a column of
ones (the intercept) in the polynomial tables, and uniform factors.
"""
import math

import torch

import paper_2211_10482_b200 as st

_FLAGS = {"f32": 0, "tf32": st.ST_FLAG_TC_TF32, "bf16": st.ST_FLAG_TC_BF16, "split": st.ST_FLAG_TC_SPLIT}
_KINDS = {"tri": st.ST_TRI_UPPER, "tet": st.ST_TET, "band": st.ST_BAND, "blockdiag": st.ST_BLOCKDIAG,
          "simplex4": st.ST_SIMPLEX4}
_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}


def listed():
    return [
        # one mini-batch of a small regression, the symmetric matrix handed to the solver: latency counts
        dict(name="cov_batch", op="moment2", mode="f32", N=4096, d=64, dense=True),
        # a table whose feature count is whatever the joins gave: rows are not even 16-byte aligned
        dict(name="cov_ragged", op="moment2", mode="f32", N=50021, d=75, dense=True),
        # many features, full fp32 arithmetic
        dict(name="cov_wide", op="moment2", mode="f32", N=65536, d=512, dense=False),
        # many features at the fp32 tolerance on the tensor cores, feature count off the tile grid
        dict(name="cov_split", op="moment2", mode="split", N=262144, d=520, dense=False),
        # the largest table: 2 GiB of bf16
        dict(name="cov_large", op="moment2", mode="bf16", N=1 << 20, d=1024, dense=False),
        # third moment of a full table in fp32
        dict(name="third_f32", op="moment3", mode="f32", N=65536, d=64),
        # third moment at reduced precision, ragged in both extents
        dict(name="third_bf16", op="moment3", mode="bf16", N=40009, d=50),
        # fourth moment (fp32 tolerance), the widest block of a degree-2 covariance
        dict(name="fourth_f32", op="moment4", mode="f32", N=30011, d=45),
        # streaming degree-2 polynomial regression: many small calls per batch
        dict(name="poly_batch", op="poly", mode="f32", N=4096, d=24),
        # factorisation kernels on structured tensors, hundreds of MB of fibres read once
        dict(name="mttkrp_cube", op="mttkrp", mode="split", I=512, K=512, R=32),
        dict(name="ttm_blocks", op="ttm", mode="tf32", kind="blockdiag", nb=64, bs=64, K=256, R=64),
        # chain in packed space, rows of an odd number of words
        dict(name="chain_tri", op="chain", kind="tri", d=384, inner=75),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _multiple(x, m):
    return max(m, x // m * m)


def _longest_K(mode, R):
    """The longest fibre drawn; on the tensor-core paths the factor has to fit in shared memory."""
    return {"f32": 1024, "tf32": min(1024, 49152 // R // 32 * 32), "split": 24576 // R // 64 * 64}[mode]


def draw(rng):
    op = rng.choice(["moment2", "moment2", "moment3", "moment4", "poly", "mttkrp", "ttm", "chain", "copy"])
    if op == "moment2":
        mode = rng.choice(["f32", "f32", "tf32", "split", "bf16"])
        d = _log(rng, 8, 1024)
        d = _multiple(d, {"f32": 1, "tf32": 4, "split": 8, "bf16": 8}[mode])
        # fp32 arithmetic: at most the listed wide table; tensor cores: at most 2^28 elements
        most = (65536 * 512 * 512 // (d * d)) if mode == "f32" else (1 << 28) // d
        return dict(op=op, mode=mode, N=_log(rng, 256, max(256, min(1 << 20, most))), d=d, dense=rng.random() < 0.5)
    if op == "moment3":
        mode = rng.choice(["f32", "tf32", "bf16"])
        d = _log(rng, 6, 112 if mode == "f32" else 64)
        return dict(op=op, mode=mode, N=_log(rng, 256, min(1 << 18, 65536 * 64 ** 3 // d ** 3)), d=d)
    if op == "moment4":
        mode = rng.choice(["f32", "bf16"])
        d = _log(rng, 4, 64)
        return dict(op=op, mode=mode, N=_log(rng, 256, min(1 << 17, 30011 * 45 ** 4 // d ** 4)), d=d)
    if op == "poly":
        return dict(op=op, mode="f32", N=_log(rng, 256, 16384), d=_log(rng, 4, 40))
    if op == "mttkrp":
        mode = rng.choice(["f32", "tf32", "split"])
        R = rng.choice([8, 16, 32, 64] if mode == "f32" else [32, 64])
        K = _multiple(_log(rng, 16, _longest_K(mode, R)), 4)
        most = math.isqrt((1 << 27) // K)           # at most 2^26 stored values
        return dict(op=op, mode=mode, I=_log(rng, 16, max(16, min(1024, most))), K=K, R=R)
    if op == "ttm":
        mode = rng.choice(["f32", "tf32", "split"])
        R = {"f32": 8 << rng.randint(0, 3), "tf32": 16 * rng.randint(1, 8), "split": 32 * rng.randint(1, 4)}[mode]
        K = _multiple(_log(rng, 16, _longest_K(mode, R)), 4)
        most = (1 << 26) // K                       # fibres
        if rng.random() < 0.5:
            bs = _log(rng, 4, 128)
            return dict(op=op, mode=mode, kind="blockdiag", nb=_log(rng, 1, max(1, min(256, most // (bs * bs)))),
                        bs=bs, K=K, R=R)
        return dict(op=op, mode=mode, kind="tri", d=_log(rng, 16, min(700, math.isqrt(2 * most) - 1)), K=K, R=R)
    if op == "chain":
        kind = rng.choice(["tri", "tet"])
        inner = _log(rng, 1, 256)
        room = (1 << 25) // inner                   # dense rows
        d = _log(rng, 16, min(2048, math.isqrt(room)) if kind == "tri" else min(160, int(room ** (1 / 3))))
        return dict(op=op, kind=kind, d=d, inner=inner)
    kind = rng.choice(["tri", "tet", "band", "blockdiag", "simplex4"])
    dtype = rng.choice(["f32", "f32", "bf16", "f64"])
    inner = rng.choice([1, _log(rng, 2, 128)])
    room = (1 << 26) // inner
    order = {"tet": 3, "simplex4": 4}.get(kind, 2)
    d = _log(rng, {2: 32, 3: 16, 4: 8}[order], min({2: 4096, 3: 256, 4: 64}[order], int(room ** (1 / order))))
    case = dict(op="copy", kind=kind, dtype=dtype, d=d, inner=inner,
                sym=kind in ("tri", "tet", "simplex4") and rng.random() < 0.7)
    if kind == "band":
        case.update(kl=rng.randint(0, d // 8), ku=rng.randint(0, d // 8))
    if kind == "blockdiag":
        bs = _log(rng, 2, max(2, d // 2))
        case.update(d=d // bs * bs, bs=bs)
    return case


def _layout(case, inner):
    kind = case["kind"]
    if kind == "blockdiag":
        bs = case["bs"]
        nb = case["nb"] if "nb" in case else case["d"] // bs
        return st.Layout(st.ST_BLOCKDIAG, nb * bs, inner, nblocks=nb, bs=bs)
    return st.Layout(_KINDS[kind], case["d"], inner, kl=case.get("kl", 0), ku=case.get("ku", 0))


def _tri(d):
    return d * (d + 1) // 2


def _tet(d):
    return d * (d + 1) * (d + 2) // 6


def _simp4(d):
    return d * (d + 1) * (d + 2) * (d + 3) // 24


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape, dtype=torch.float32):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device="cuda").mul_(2).sub_(1)

    op = case["op"]
    s = dict(op=op, flags=_FLAGS.get(case.get("mode", "f32"), 0))
    if op == "moment2":
        bf16 = case["mode"] == "bf16"
        s["flags"] = 0 if bf16 else s["flags"]      # a bf16 table selects its own path
        s["X"] = normal(case["N"], case["d"], dtype=torch.bfloat16 if bf16 else torch.float32)
        s["layout"] = st.Layout(st.ST_TRI_UPPER, case["d"]) if case["dense"] else None
    elif op in ("moment3", "moment4"):
        s["X"] = normal(case["N"], case["d"])
    elif op == "poly":
        d = case["d"]
        s["X"] = normal(case["N"], d)
        s["X"][:, 0] = 1.0
        s["sums"] = tuple(normal(n).mul_(case["N"]) for n in (_tri(d), _tet(d), _simp4(d)))
    elif op == "mttkrp":
        s["B"] = uniform(_tri(case["I"]), case["K"])
        s["C"] = uniform(case["I"], case["R"])
        s["D"] = uniform(case["K"], case["R"])
    elif op == "ttm":
        K = case["K"]
        s["layout"] = _layout(case, K)
        s["blocks"] = (case["nb"], case["bs"]) if case["kind"] == "blockdiag" else None
        s["B"] = normal(st.st_packed_elems(s["layout"]) // K, K)
        s["U"] = normal(K, case["R"])
    elif op == "chain":
        s["layout"] = _layout(case, case["inner"])
        s["dense"] = normal(st.st_dense_elems(s["layout"]))
        s["B"] = normal(st.st_packed_elems(s["layout"]))
        s["E"] = normal(st.st_dense_elems(s["layout"]))
    else:
        s["layout"] = _layout(case, case["inner"])
        s["dense"] = normal(st.st_dense_elems(s["layout"]), dtype=_DTYPES[case["dtype"]])
        s["fill"] = st.ST_FILL_SYMMETRIC if case["sym"] else st.ST_FILL_ZERO
    return s


def run(s):
    op, flags = s["op"], s["flags"]
    if op == "moment2":
        packed = st.st_sym_moment2(s["X"], flags=flags)
        if s["layout"] is None:
            return packed
        return packed, st.st_unpack(packed, s["layout"], st.ST_FILL_SYMMETRIC)
    if op == "moment3":
        return st.st_sym_moment3(s["X"], flags=flags)
    if op == "moment4":
        return st.st_sym_moment4(s["X"], flags=flags)
    if op == "poly":
        X, (a, b, c) = s["X"], s["sums"]
        return (st.st_packed_axpby(0.99, a, 1.0, st.st_sym_moment2(X)),
                st.st_packed_axpby(0.99, b, 1.0, st.st_sym_moment3(X)),
                st.st_packed_axpby(0.99, c, 1.0, st.st_sym_moment4(X)))
    if op == "mttkrp":
        return st.st_mttkrp_tri(s["B"], s["C"], s["D"], flags=flags)
    if op == "ttm":
        if s["blocks"] is not None:
            return st.st_ttm_blockdiag(s["B"], s["U"], *s["blocks"], flags=flags)
        return st.st_ttm_packed(s["B"], s["U"], s["layout"], flags=flags)
    if op == "chain":
        layout = s["layout"]
        product = st.st_thp(s["B"], s["dense"], layout)
        total = st.st_packed_axpby(1.0, product, 0.5, st.st_pack(s["E"], layout))
        return st.st_unpack(total, layout, st.ST_FILL_SYMMETRIC)
    packed = st.st_pack(s["dense"], s["layout"])
    return packed, st.st_unpack(packed, s["layout"], s["fill"])


def work(case):
    """Bytes: every input read once, every output written once.  Flops: the unique terms only, products
    shared between terms counted once."""
    op = case["op"]
    if op in ("moment2", "moment3", "moment4", "poly"):
        N, d = case["N"], case["d"]
        out = {"moment2": _tri(d), "moment3": _tet(d), "moment4": _simp4(d)}
        flops = {"moment2": 2 * N * _tri(d), "moment3": N * (2 * _tet(d) + _tri(d)),
                 "moment4": N * (2 * _simp4(d) + _tri(d))}
        if op == "poly":
            return {"bytes": 4 * (N * d + 2 * sum(out.values())), "flops": sum(flops.values())}
        es = 2 if op == "moment2" and case["mode"] == "bf16" else 4
        dense = 4 * d * d if case.get("dense") else 0
        return {"bytes": es * N * d + 4 * out[op] + dense, "flops": flops[op]}
    if op == "mttkrp":
        I, K, R = case["I"], case["K"], case["R"]
        return {"bytes": 4 * (_tri(I) * K + (2 * I + K) * R), "flops": 2 * R * _tri(I) * (K + 1)}
    if op == "ttm":
        rows = case["nb"] * case["bs"] ** 2 if case["kind"] == "blockdiag" else _tri(case["d"])
        K, R = case["K"], case["R"]
        return {"bytes": 4 * (rows * (K + R) + K * R), "flops": 2 * rows * K * R}
    layout = _layout(case, case["inner"])
    packed, dense = st.st_packed_elems(layout), st.st_dense_elems(layout)
    if op == "chain":                   # B, the unique part of the two dense operands, the dense result
        return {"bytes": 4 * (3 * packed + dense), "flops": 4 * packed}
    es = {"f32": 4, "bf16": 2, "f64": 8}[case["dtype"]]
    return {"bytes": es * (2 * packed + dense), "flops": 0}


# (relative 2-norm error, largest error over the result's root mean square or value): about four times what
# the calls show against the same sums in fp64, over the listed cases and 150 drawn ones.  tf32 truncates
# its operands, so sums of squares come out low by up to 2^-10 relative.
_TOLERANCE = {
    ("moment2", "f32"): (2e-6, 8e-6), ("moment2", "tf32"): (3e-3, 4e-3), ("moment2", "split"): (5e-5, 6e-5),
    ("moment2", "bf16"): (7e-6, 1e-5),
    ("moment3", "f32"): (2e-6, 1.5e-5), ("moment3", "tf32"): (2.4e-3, 2e-2), ("moment3", "bf16"): (1.2e-2, 7e-2),
    ("moment4", "f32"): (7e-5, 8e-5), ("moment4", "bf16"): (2e-3, 3e-3), ("poly", "f32"): (8e-6, 1.4e-4),
    ("mttkrp", "f32"): (1.6e-6, 8e-6), ("mttkrp", "tf32"): (1.7e-3, 7e-3), ("mttkrp", "split"): (1.6e-5, 9e-5),
    ("ttm", "f32"): (5e-7, 2e-6), ("ttm", "tf32"): (2e-3, 9e-3), ("ttm", "split"): (1.8e-5, 1.3e-4),
    ("chain", None): (5e-7, 1e-6),
}


def tolerance(case):
    if case["op"] == "copy":
        return "exact"
    rel, most = _TOLERANCE[case["op"], case.get("mode")]
    return {"rel": rel, "max": most}
