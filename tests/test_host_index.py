"""CPU tests of the library's host logic: closed-form index arithmetic against the oracle's
running-counter walk, the exported symbols, and host-side argument validation."""
import ctypes
import os
import re
import subprocess
import tempfile

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_10482_b200", "csrc")


@pytest.fixture(scope="module")
def shim():
    out = os.path.join(tempfile.mkdtemp(prefix="st_shim_"), "shim.so")
    subprocess.check_call(["g++", "-O2", "-shared", "-fPIC", "-std=c++17", "-x", "c++", "-I", CSRC,
                           os.path.join(ROOT, "tests", "index_host_shim.cpp"), "-o", out])
    L = ctypes.CDLL(out)
    ll = ctypes.c_longlong
    for name in ("shim_tri_rows", "shim_tet_rows", "shim_check_all_tri", "shim_check_all_tet", "shim_simp4_rows",
                 "shim_check_all_simp4"):
        getattr(L, name).argtypes = [ll]
        getattr(L, name).restype = ll
    L.shim_tri_encode.argtypes = [ll, ll, ll]
    L.shim_tri_encode.restype = ll
    L.shim_tet_encode.argtypes = [ll, ll, ll, ll]
    L.shim_tet_encode.restype = ll
    L.shim_tri_decode.argtypes = [ll, ll, ctypes.POINTER(ll), ctypes.POINTER(ll)]
    L.shim_tet_decode.argtypes = [ll, ll, ctypes.POINTER(ll), ctypes.POINTER(ll), ctypes.POINTER(ll)]
    return L


def test_closed_forms_match_the_oracle_walk(shim):
    for d in list(range(1, 13)) + [17, 31]:
        assert shim.shim_tri_rows(d) == oracle.packed_rows(oracle.KIND_TRI, d)
        assert shim.shim_tet_rows(d) == oracle.packed_rows(oracle.KIND_TET, d)
    for d in (1, 2, 5, 9):
        for i in range(d):
            for j in range(i, d):
                assert shim.shim_tri_encode(d, i, j) == oracle.locate(oracle.KIND_TRI, d, i, j)
                for k in range(j, d):
                    assert shim.shim_tet_encode(d, i, j, k) == oracle.locate(oracle.KIND_TET, d, i, j, k)


def test_decode_is_exact_for_every_position(shim):
    for d in range(1, 49):
        assert shim.shim_check_all_tri(d) == 0
        assert shim.shim_check_all_tet(d) == 0
    for d in (64, 100, 257):
        assert shim.shim_check_all_tet(d) == 0
    for d in (1000, 1024, 4097):
        assert shim.shim_check_all_tri(d) == 0


def test_four_simplex_positions_and_the_count_the_paper_gives(shim):
    # Section 2, "Intricate Structures": the degree-2 polynomial-regression covariance on 4 features has
    # 65 distinct elements = 10 (pairs) + 20 (triples) + 35 (4-tuples with repetition)
    assert shim.shim_tri_rows(4) + shim.shim_tet_rows(4) + shim.shim_simp4_rows(4) == 65
    assert shim.shim_simp4_rows(4) == 35
    for d in list(range(1, 20)) + [33, 64]:
        assert shim.shim_check_all_simp4(d) == 0


def test_decode_at_boundaries_of_large_extents(shim):
    ll = ctypes.c_longlong
    rng = np.random.default_rng(5)
    for d in (1 << 16, (1 << 20) - 3, 1 << 20, (1 << 31) - 1):
        rows = [0, 1, d // 2, d - 2, d - 1] + [int(x) for x in rng.integers(0, d, 20)]
        for i in rows:
            for j in (i, min(i + 1, d - 1), d - 1):
                p = shim.shim_tri_encode(d, i, j)
                a, b = ll(), ll()
                shim.shim_tri_decode(d, p, ctypes.byref(a), ctypes.byref(b))
                assert (a.value, b.value) == (i, j)
        assert shim.shim_tri_encode(d, d - 1, d - 1) == shim.shim_tri_rows(d) - 1
    for d in (1 << 10, 50000, 1 << 20):
        rows = [0, 1, d // 3, d - 2, d - 1] + [int(x) for x in rng.integers(0, d, 10)]
        for i in rows:
            for j in (i, (i + d) // 2, d - 1):
                for k in (j, d - 1):
                    q = shim.shim_tet_encode(d, i, j, k)
                    a, b, c = ll(), ll(), ll()
                    shim.shim_tet_decode(d, q, ctypes.byref(a), ctypes.byref(b), ctypes.byref(c))
                    assert (a.value, b.value, c.value) == (i, j, k)
        assert shim.shim_tet_encode(d, d - 1, d - 1, d - 1) == shim.shim_tet_rows(d) - 1


# ---------------------------------------------------------------- the C ABI library itself

def _declared():
    text = open(os.path.join(ROOT, "include", "structtensor.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(st_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    import paper_2211_10482_b200 as st
    from paper_2211_10482_b200 import _build
    _build.build()
    L = ctypes.CDLL(st.LIB_PATH)
    names = _declared()
    assert len(names) >= 12
    for n in names:
        assert hasattr(L, n), n
    assert sorted(st.EXPORTS) == names
    assert st.lib().st_abi_version() == 1
    assert st.status_string(st.ST_ERR_WORKSPACE) == "workspace missing or too small"


def test_layout_sizes_and_host_side_validation():
    import paper_2211_10482_b200 as st
    L = st.lib()
    assert st.st_packed_elems(st.Layout(st.ST_TRI_UPPER, 64)) == 2080
    assert st.st_packed_elems(st.Layout(st.ST_TET, 64)) == 45760
    assert st.st_packed_elems(st.Layout(st.ST_TRI_UPPER, 512, inner=512)) == 67239936
    assert st.st_packed_elems(st.Layout(st.ST_BLOCKDIAG, 4096, inner=256, nblocks=64, bs=64)) == 67108864
    assert st.st_packed_elems(st.Layout(st.ST_BAND, 10, kl=2, ku=1)) == 40
    assert st.st_packed_elems(st.Layout(st.ST_BLOCKDIAG, 10, nblocks=3, bs=3)) == -1
    assert st.st_packed_elems(st.Layout(st.ST_TRI_UPPER, 0)) == -1
    assert st.st_packed_elems(st.Layout(7, 4)) == -1
    assert st.st_dense_elems(st.Layout(st.ST_TET, 5, inner=2)) == 250
    for kind, kw in ((st.ST_TRI_UPPER, {}), (st.ST_TET, {}), (st.ST_BAND, dict(kl=1, ku=2)),
                     (st.ST_BLOCKDIAG, dict(nblocks=2, bs=3))):
        lay = st.Layout(kind, 6, inner=3, **kw)
        okw = {("nb" if k == "nblocks" else k): v for k, v in kw.items()}
        assert st.st_packed_elems(lay) == 3 * oracle.packed_rows(kind, 6, **okw)
    # argument errors are reported before anything touches a device
    lay = st.Layout(st.ST_TRI_UPPER, 4).c()
    assert L.st_pack(ctypes.byref(lay), st.ST_F32, None, None, None) == st.ST_ERR_NULL
    assert L.st_pack(ctypes.byref(lay), st.ST_F32, 256, 8, None) == st.ST_ERR_ALIGN
    assert L.st_pack(ctypes.byref(lay), 9, 256, 512, None) == st.ST_ERR_DTYPE
    bad = st.Layout(st.ST_BLOCKDIAG, 7, nblocks=2, bs=3).c()
    assert L.st_unpack(ctypes.byref(bad), st.ST_F32, 256, 512, 0, None) == st.ST_ERR_SHAPE
    band = st.Layout(st.ST_BAND, 7, kl=1, ku=1).c()
    assert L.st_unpack(ctypes.byref(band), st.ST_F32, 256, 512, st.ST_FILL_SYMMETRIC, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_sym_moment2(None, st.ST_F32, 4, 4, 4, 256, None, 0, 0, None) == st.ST_ERR_NULL
    assert L.st_sym_moment2(256, st.ST_F32, 4, 4, 3, 512, None, 0, 0, None) == st.ST_ERR_SHAPE
    assert L.st_sym_moment2(256, st.ST_F64, 4, 4, 4, 512, None, 0, 0, None) == st.ST_ERR_DTYPE
    assert L.st_sym_moment2(256, st.ST_F32, 4, 4, 4, 512, None, 0, 0, None) == st.ST_ERR_WORKSPACE
    assert L.st_sym_moment3(256, 4, 257, 257, 512, None, 0, 0, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_sym_moment3(264, 4, 16, 16, 512, None, 0, 0, None) == st.ST_ERR_ALIGN
    # fp32 takes any feature count, dense control too, also where one of its routes has no plan
    for d in (3068, 3072, 3076, 4096, 4100):
        for flags in (0, st.ST_FLAG_DENSE_CONTROL):
            assert L.st_sym_moment2(256, st.ST_F32, 260, d, d, 512, None, 0, flags, None) == st.ST_ERR_WORKSPACE, (d, flags)
    assert L.st_sym_moment3(256, 4, 16, 16, 512, None, 0, 0, None) == st.ST_ERR_WORKSPACE
    assert L.st_sym_moment3(256, 4, 12, 18, 512, None, 0, 0, None) == st.ST_ERR_WORKSPACE     # any d, any pitch
    assert L.st_sym_moment3(256, 4, 72, 72, 512, None, 0, st.ST_FLAG_TC_TF32, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_sym_moment3(256, 4, 13, 13, 512, None, 0, st.ST_FLAG_TC_BF16, None) == st.ST_ERR_WORKSPACE
    assert L.st_sym_moment4(256, 4, 129, 129, 512, None, 0, 0, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_sym_moment4(256, 4, 8, 8, 512, None, 0, 0, None) == st.ST_ERR_WORKSPACE
    assert L.st_mttkrp_tri(256, 4, 8, 512, 768, 12, 1024, None, 0, 0, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_mttkrp_tri(256, 4, 8, 512, 768, 0, 1024, None, 0, 0, None) == st.ST_ERR_SHAPE
    assert L.st_ttm_blockdiag(256, 2, 2, 8, 512, 24, 1024, None, 0, 0, None) == st.ST_ERR_UNSUPPORTED
    assert L.st_ttm_blockdiag(256, 2, 2, 8, 520, 32, 1024, None, 0, 0, None) == st.ST_ERR_ALIGN
    assert st.st_workspace_bytes(st.ST_OP_SYM_MOMENT3, 65536, 64) > 45760 * 4
    assert st.st_workspace_bytes(st.ST_OP_SYM_MOMENT3, 65536, 63) > 41664 * 4
    assert st.st_workspace_bytes(st.ST_OP_SYM_MOMENT3, 65536, 257) == 0
    # beyond 64 features the tile table of the call lives in the workspace too
    assert st.st_workspace_bytes(st.ST_OP_SYM_MOMENT3, 100, 128) > 128 * 129 * 130 // 6 * 4 + 6528 * 4
    assert st.st_workspace_bytes(st.ST_OP_SYM_MOMENT2, 4096, 64, st.ST_F32) >= 256


def test_kernels_do_not_read_through_the_read_only_path():
    # Every kernel is launched as a programmatic dependent: its blocks may be there while its input is still being written.
    # ld.global.nc, __ldg and what a compiler makes of `const T *__restrict__` kernel parameters are for data that is
    # read-only for as long as the kernel lives.
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        found += [(name, w) for w in re.findall(r"__ldg\s*\(|ld\.global(?:\.\w+)*\.nc", text)]
        for head in re.findall(r"__global__[^{;]*\{", text):
            found += [(name, w) for w in re.findall(r"const\s+[\w:<> ]+\*\s*__restrict__", head)]
        found += [(name, w) for w in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s*\w+\s*=\s*a\.", text)]
    assert not found, found


def test_sizes_that_leave_64_bits_do_not_match_by_wrapping_around():
    import torch
    import paper_2211_10482_b200 as st
    B, U = torch.zeros(4), torch.zeros(4, 8)
    for nb, bs in ((2 ** 62 + 1, 1), (-(2 ** 62) + 1, 1), (-1, -1)):        # nb bs bs 4 = 4 modulo 2^64; two signs that cancel
        with pytest.raises(ValueError, match="shape mismatch"):
            st.st_ttm_blockdiag(B, U, nb, bs)
    with pytest.raises(ValueError, match="shape mismatch"):                 # (2^32)^2 = 0 modulo 2^64
        st.st_ttm_blockdiag(torch.zeros(0), U, 2 ** 32, 1, flags=st.ST_FLAG_DENSE_CONTROL)
    with pytest.raises(ValueError, match="shape mismatch"):
        st.st_mttkrp_tri(torch.zeros(0), torch.zeros(2 ** 33, 0), torch.zeros(4, 0))


def test_a_fill_is_whatever_int_makes_of_it():
    import torch
    import paper_2211_10482_b200 as st
    packed, lay = torch.zeros(6), st.Layout(st.ST_TRI_UPPER, 3)
    for fill in (1, 1.0, "1", True, np.int64(1)):
        with pytest.raises(ValueError, match="CUDA"):                       # accepted: the host tensor is what is refused
            st.st_unpack(packed, lay, fill)
    for fill in (None, "x", 1j):
        with pytest.raises((TypeError, ValueError), match="int"):
            st.st_unpack(packed, lay, fill)


def test_arrivals_at_another_block_name_the_scope_of_the_cluster():
    # An arrival orders nothing for another block's threads unless its scope, or that of a fence before a relaxed one, is the
    # cluster's; without one it is that of the block.
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"mbarrier\.arrive[\w.:]*shared::cluster", text):
            if ".release.cluster" in m.group():
                continue
            if ".relaxed.cluster" not in m.group() or "fence.release.sync_restrict::shared::cta.cluster" not in text[max(0, m.start() - 200):m.start()]:
                found.append((name, m.group()))
    assert not found, found


def test_the_one_launch_second_moment_is_taken_where_clusters_fit_and_it_was_measured_to_be_faster():
    src = os.path.join(tempfile.mkdtemp(prefix="st_rule_"), "rule.cpp")
    with open(src, "w") as f:
        f.write('#include "moment2_rule.cuh"\nextern "C" int rule(long long N, int items, int clusters, int rg, int bulk, int fit)\n'
                "{ return st::m2s_use_cluster(N, items, clusters, rg, bulk != 0, fit); }\n")
    subprocess.check_call(["g++", "-shared", "-fPIC", "-std=c++17", "-I", CSRC, src, "-o", src + ".so"])
    rule = ctypes.CDLL(src + ".so").rule
    rule.argtypes = [ctypes.c_longlong] + [ctypes.c_int] * 5

    def use(N, d, fit=8):                                        # items, clusters and row groups as the plan makes them
        nbk = (d + 7) // 8
        items = (nbk * (nbk + 1) // 2 + 1) // 2
        clusters = (items + 4) // 5
        per = (items + clusters - 1) // clusters
        rg = min(128 // per, 57344 // (4 * ((d + 3) // 4 * 4)) // 8)
        return rule(N, items, (items + per - 1) // per, rg, d % 4 == 0, fit)

    for N, d in ((32, 8), (16384, 8), (8192, 16), (4096, 24), (8000, 64), (1, 100), (4096, 100), (3000, 120), (2000, 33), (1000, 75)):
        assert use(N, d) and not use(N, d, fit=0), (N, d)        # no cluster fits: the two launches
    for N, d in ((30000, 8), (16384, 16), (6000, 24), (16384, 64), (6000, 100), (4096, 120), (3000, 33), (2000, 75)):
        assert not use(N, d), (N, d)


def test_the_binding_belongs_to_either_build_and_to_one_python_and_torch(tmp_path, monkeypatch):
    from paper_2211_10482_b200 import _build
    for name in ("OBJDIR", "OBJDIR_CHECK", "LIB", "LIB_CHECK", "BINDING"):
        monkeypatch.setattr(_build, name, str(tmp_path / name))
    monkeypatch.setattr(_build, "BINDING_KEY", str(tmp_path / "key"))
    monkeypatch.setattr(_build, "_sources", lambda: [])
    made = []

    def run(cmd, **kw):
        made.append(cmd[0])
        open(cmd[cmd.index("-o") + 1], "w").close()
        return subprocess.CompletedProcess(cmd, 0, "", "")

    monkeypatch.setattr(_build.subprocess, "run", run)
    _build.build(check=True)
    assert made == ["g++", "nvcc"] or made == ["nvcc", "g++"]
    _build.build(check=True)
    _build._build_binding(False)
    assert len(made) == 2                                        # up to date
    monkeypatch.setattr(_build, "_binding_key", lambda: "another torch")
    _build._build_binding(False)
    assert made[2:] == ["g++"]


def test_fourth_moment_in_bf16_takes_as_many_samples_as_its_copies_can_name():
    import paper_2211_10482_b200 as st
    size = lambda N: st.st_workspace_bytes(st.ST_OP_SYM_MOMENT4, N, 4, 0, 0, st.ST_FLAG_TC_BF16)
    for N in (1 << 29, (1 << 29) + 1, (1 << 31) - 64):
        assert size(N) > N * 10 * 2, N                           # ten pair features a sample
    assert size((1 << 31) - 63) == 0


def test_a_workspace_for_more_samples_serves_fewer_on_the_tensor_cores():
    """Second moment in bf16, TF32 and split: columns that many samples carry along have tiles of their own with few."""
    import paper_2211_10482_b200 as st
    modes = ((st.ST_BF16, 0, 8), (st.ST_F32, st.ST_FLAG_TC_TF32, 4), (st.ST_F32, st.ST_FLAG_TC_SPLIT, 8))
    samples = sorted({1, 33, 66, 128} | {500 * i for i in range(1, 200)} | {1 << k for k in range(10, 29)})
    for dtype, flags, step in modes:
        for d in sorted({256 * k + step * c for k in range(1, 16) for c in (1, 2, 5, 9, 128 // step)} | {824, 1800, 4096}):
            sizes = [st.st_workspace_bytes(st.ST_OP_SYM_MOMENT2, N, d, dtype, 0, flags) for N in samples]
            assert sizes == sorted(sizes), (flags, d)


def test_copies_read_no_byte_behind_the_source_array():
    src = os.path.join(tempfile.mkdtemp(prefix="st_span_"), "span.cpp")
    with open(src, "w") as f:
        f.write("""#include "copy_span.cuh"
// runs [x, x + n) of an array of `size` bytes on a 16-byte boundary, to every offset: what is read stays inside, every byte is
// copied once, and at most the last unit goes singly
extern "C" long long bad(int size, int es)
{
    long long bad = 0;
    const uintptr_t base = 4096, end = base + size;
    for (int to = 0; to < 16; to += es)
        for (int x = 0; x < size; x += es)
            for (int n = es; x + n <= size; n += es) {
                const st::CopySpan c = st::copy_span(8192 + to, base + x, n, end);
                const uintptr_t first = base + x + c.head, last = first - c.off + 16 * (uintptr_t)(c.units + (c.off ? 1 : 0));
                bad += c.units > 0 && (last > (end + (c.off ? 0 : 15)) || first - c.off < base);
                bad += c.units > 0 && !c.off && first + 16 * (uintptr_t)c.units > end;
                bad += c.units > 0 && (8192 + to + c.head) % 16 != 0;
                bad += c.units < 0 || c.head + 16 * c.units > n || c.ends != n - 16 * c.units || c.ends % es || c.ends >= 48;
            }
    return bad;
}
""")
    subprocess.check_call(["g++", "-O2", "-shared", "-fPIC", "-std=c++17", "-I", CSRC, src, "-o", src + ".so"])
    L = ctypes.CDLL(src + ".so")
    L.bad.restype = ctypes.c_longlong
    for es in (2, 4, 8):
        for size in range(es, 160, es):
            assert L.bad(size, es) == 0, (size, es)
