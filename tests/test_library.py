"""The C-ABI library builds, loads without a GPU and exports every symbol the header declares; the binding's
structs match the header's layout."""
import ctypes as C
import os
import re
import subprocess

import pytest

from paper_2501_14183_b200 import binding as vd
from paper_2501_14183_b200 import build as lib_build
from util import RADIX_LENGTHS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = []
    inc = os.path.join(ROOT, "include")
    for fn in sorted(os.listdir(inc)):
        if not fn.endswith(".h"):
            continue
        text = open(os.path.join(inc, fn)).read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        names += re.findall(r"\b(vardrop_[a-z0-9_]+)\s*\(", text)
    return sorted(set(names))


@pytest.fixture(scope="module")
def lib():
    lib_build.build()
    return vd.load()


def test_exports_every_declared_symbol(lib):
    names = declared_functions()
    assert {"vardrop_hash", "vardrop_select", "vardrop_attn_fwd", "vardrop_attn_bwd"} <= set(names)
    for name in names:
        assert hasattr(lib, name), name
    assert set(names) == set(vd.EXPORTS)


def test_status_strings_and_version(lib):
    assert lib.vardrop_version().decode().count(".") == 1
    texts = [lib.vardrop_status_string(i).decode() for i in range(7)]
    assert texts[0] == "ok" and len(set(texts)) == 7
    assert lib.vardrop_status_string(99).decode() == "unknown status"


def test_struct_layouts_match_header():
    assert C.sizeof(vd.HashCfg) == 28
    assert C.sizeof(vd.SelectCfg) == 40 and vd.SelectCfg.rate.offset == 16 and vd.SelectCfg.seed.offset == 24
    assert C.sizeof(vd.AttnCfg) == 48 and vd.AttnCfg.sB.offset == 24


def test_workspace_queries_need_no_gpu(lib):
    assert vd.vardrop_hash_workspace_bytes(vd.HashCfg(32, 321, 96, 3, 0, 0, 0)) >= 4
    s1 = vd.vardrop_select_workspace_bytes(vd.SelectCfg(1, 321, 0, 0.3, 1, 0))
    s2 = vd.vardrop_select_workspace_bytes(vd.SelectCfg(4, 321, 0, 0.3, 1, 0))
    assert 0 < s1 < s2
    assert vd.vardrop_select_workspace_bytes(vd.SelectCfg(1, 0, 0, 0.3, 1, 0)) == 0          # invalid config
    a = vd.vardrop_attn_workspace_bytes(vd.AttnCfg(32, 321, 8, 64, 0.0))
    assert a > 4 * 32 * 384 * 8 * 128
    assert vd.vardrop_attn_workspace_bytes(vd.AttnCfg(32, 321, 8, 128, 0.0)) == 0            # unsupported head dim


def test_host_side_validation_needs_no_gpu(lib):
    # argument checks run before any CUDA call: bad configs are rejected on a machine without a GPU too
    st = lib.vardrop_hash(None, C.byref(vd.HashCfg(2, 4, 8200, 3, 0, 0, 0)), None, None, None, None, 0, None)
    assert st == vd.ERR_UNSUPPORTED and b"above 8192" in lib.vardrop_last_error()
    st = lib.vardrop_hash(None, C.byref(vd.HashCfg(2, 4, 96, 3, 0, 0, 0)), None, None, None, None, 0, None)
    assert st == vd.ERR_INVALID_ARG and b"x is NULL" in lib.vardrop_last_error()
    st = lib.vardrop_attn_fwd(None, None, None, None, None, C.byref(vd.AttnCfg(1, 8, 1, 48, 0.0)), None, None, None, 0, None)
    assert st == vd.ERR_UNSUPPORTED


def kernel_bodies():
    """(file, name, text without comments) of every __global__ function."""
    csrc = os.path.join(ROOT, "paper_2501_14183_b200", "csrc")
    for fn in sorted(os.listdir(csrc)):
        if not fn.endswith(".cu"):
            continue
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(csrc, fn)).read(), flags=re.S)
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\([^{;]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield fn, m.group(1), text[m.end():end]


def test_peers_shared_memory_is_reached_behind_a_cluster_barrier():
    """A CTA's shared memory may only be reached from another one of its cluster once it runs, which nothing but a barrier of the cluster says: in the
    text of a kernel one is waited for ahead of the first remote access."""
    seen = []
    for fn, name, body in kernel_bodies():
        remote = re.search(r"\bpeer_(addr|store\d)\s*\(|\bfirst_cta_addr\s*\(|(ld|st|red|atom)\.shared::cluster", body)
        if not remote:
            continue
        seen.append(name)
        barrier = re.search(r"\bcluster_(sync|wait)\s*\(\)", body)
        assert barrier and barrier.start() < remote.start(), f"{fn}: {name}"
    assert set(seen) == {"select_cluster_kernel", "hash_dft_kernel"}


@pytest.fixture(scope="module")
def plan_lib(tmp_path_factory):
    """The host-side plan of the transform, which is plain C++."""
    d = tmp_path_factory.mktemp("plan")
    src = d / "plan.cpp"
    src.write_text('#include "hash_plan.h"\nusing namespace vardrop;\n'
                   'static int put(const RadixPlan& p, int* r) { for (int i = 0; i < p.n; ++i) r[i] = p.radix[i]; return p.n; }\n'
                   'extern "C" int plan(int L, int* r, int* wide, int* sums) { RadixPlan p = radix_plan(L); *wide = p.wide; *sums = p.sums; return put(p, r); }\n'
                   'extern "C" int narrow(int L, int* r) { return put(fours_and_primes(L), r); }\n'
                   'extern "C" int threads(int L, int n, int rows, int ctas, int smem, int few, int sms) { return hash_threads(radix_plan(L), L, n, rows, ctas, smem, few, sms); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{ROOT}/paper_2501_14183_b200/csrc", "-o", str(d / "plan.so"), str(src)])
    return C.CDLL(str(d / "plan.so"))


def radix_plans(plan_lib, longest=8192):
    for L in range(2, longest + 1):
        r, n, wide, sums = (C.c_int * 16)(), (C.c_int * 16)(), C.c_int(), C.c_int()
        count = plan_lib.plan(L, r, C.byref(wide), C.byref(sums))
        yield L, list(r[:count]), list(n[:plan_lib.narrow(L, n)]), bool(wide.value), bool(sums.value)


def test_radix_plan_of_every_length(plan_lib):
    """The product of the radices is the length; radices 6 and 8 to 10, which cost every call of their kernel registers, only where they save a stage; no
    two-point stage where a four and a four do as well as an eight and a two; not two eights, slower and less exact than three fours."""
    for L, radices, narrow, wide, sums in radix_plans(plan_lib):
        prod = 1
        for r in radices:
            prod *= r
        assert prod == L, L
        assert wide == any(r in (6, 8, 9, 10) for r in radices), L
        assert len(radices) < len(narrow) if wide else radices == narrow, (L, radices, narrow)
        assert not (8 in radices and 2 in radices) and radices != [8, 8], (L, radices)
        assert sums == (radices[-1] > 10), L


def test_threads_of_the_transform(plan_lib):
    """The threads of a CTA go by the stage with the most butterflies (the first, of the largest radix, has the fewest), by the rounds that the CTAs take, and not
    by a last radix above 7, which is no stage of plain sums."""
    sms, kb = 148, 20 * 1024
    threads = lambda L, transforms, rows, ctas, smem, few: plan_lib.threads(L, transforms, rows, ctas, smem, few, sms)  # noqa: E731
    assert threads(960, 1, 1, 100, kb, 1) == 512 and threads(1024, 1, 1, 100, kb, 1) == 256          # 8 8 3 5: 320 butterflies; 8 8 4 4: 256
    assert threads(300, 1, 1, 100, kb, 1) == 128 and threads(1000, 1, 1, 100, kb, 1) == 256          # 10 6 5: 60; 10 10 10: 100
    assert threads(90, 8, 1, 862, kb, 0) == 128 and threads(112, 8, 1, 1000, kb, 0) == 128           # one round, where 256 threads take two
    assert threads(1000, 2, 1, 862, 2 * kb, 0) == 256 and threads(384, 4, 2, 1250, 28 * 1024, 0) == 256     # two rounds of either
    for L, radices, _, wide, sums in radix_plans(plan_lib, 1024):
        most = max(L if r > 10 else L // r for r in radices)
        for transforms in (1, 2, 8):
            for ctas in (30, 200, 500, 700, 1000, 5000):
                t = threads(L, transforms, 1, ctas, kb, int(ctas < 2 * sms))
                assert t in (128, 256, 512) and (t < 512 or ctas <= 2 * sms)
                if wide and ctas <= 2 * sms:
                    assert min(512, transforms * most) / 2 <= t <= max(128, 4 * transforms * most), (L, transforms, ctas, t)


def test_radix_lengths_cover_every_radix_at_every_place(plan_lib):
    """Lengths with a prime factor above 7 do not count: the matrix product may take them."""
    places = set()
    for L, radices, _, _, sums in radix_plans(plan_lib, 4000):
        if L in RADIX_LENGTHS and not sums and len(radices) > 1:
            places |= {(radices[0], "first"), (radices[-1], "last")} | {(r, "middle") for r in radices[1:-1]}
    assert places == {(r, at) for r in range(2, 11) for at in ("first", "middle", "last")}
