"""The C-ABI library builds, loads without a GPU and exports every symbol the header declares; the binding's
structs match the header's layout."""
import ctypes as C
import os
import re
import subprocess

import numpy as np
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


# What the branch of bwd_many_kernel that takes results out needs around it to run on the host, a thread a warp: waits that succeed but for one, and a named
# barrier that says when not all four come.
HOST_WARPGROUP = r"""
#include <chrono>
#include <condition_variable>
#include <cstdint>
#include <mutex>
#include <thread>
struct uint4 { uint32_t x, y, z, w; };
struct float4 { float x, y, z, w; };
typedef uint16_t __nv_bfloat16;
struct CUtensorMap {};
struct Item { int jt, h, b, n_sel; };
struct Params { __nv_bfloat16 *k, *v, *dk, *dv; const int32_t *sel_idx, *n_sel; long long sB, sN, sH; int B, N, H, D, S; float scale; } P;
const int kTile = 128, kRowBytes = 128, kTileBytes = 16384;
const uint32_t kColDq = 0, kColDv = 0, kColDk = 0;
alignas(16) unsigned char buf_smem[8 * 16384];
unsigned char *sK = buf_smem, *sV = buf_smem + 2 * kTileBytes, *sOut = buf_smem + 4 * kTileBytes;
CUtensorMap map_acc;
const Item items[5] = {{0, 0, 0, 300}, {1, 0, 0, 100}, {0, 1, 0, 200}, {0, 0, 0, -1}, {0, 0, 0, -1}};
std::mutex m;
std::condition_variable cv;
int arrived, gone, phase, waits[4], fail_warp, fail_at;
bool all_ok, result, hung;
thread_local int me;
bool group_sync_and(int, bool ok) {
    std::unique_lock<std::mutex> l(m);
    all_ok = (arrived ? all_ok : true) && ok;
    const int p = phase;
    if (++arrived == 4) { arrived = 0; ++phase; result = all_ok; cv.notify_all(); return result; }
    cv.notify_all();
    cv.wait(l, [&] { return phase != p || hung || arrived + gone == 4; });      // the last says that no more will come
    if (phase == p) { hung = true; cv.notify_all(); return false; }
    return result;
}
bool warp_wait_relaxed(uint64_t*, uint32_t) { return !(me == fail_warp && waits[me]++ == fail_at); }
template <class T> T __ldg(const T* p) { return *p; }
uint32_t pack2(float, float) { return 0; }
uint4 make_uint4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) { return {a, b, c, d}; }
float4 make_float4(float a, float b, float c, float d) { return {a, b, c, d}; }
template <class... A> void nothing(A&&...) {}
#define bulk_wait_group_read0 nothing
#define bulk_wait_group0 nothing
#define bulk_commit_group nothing
#define tma_reduce_add_4d nothing
#define copy_32_picked nothing
#define cp_async_arrive nothing
#define tc_fence_after nothing
#define tc_fence_before nothing
#define tmem_ld32(at, v) for (float& e : v) e = 0.f
#define tmem_ld_wait nothing
#define fence_proxy_async_smem nothing
template <bool kRows> void role(int warp, bool& left_ok) {
    const int lane = 0, tid = warp * 32;
    uint32_t tmem = 0;
    bool ok = true;
    uint64_t bars[64];
    uint64_t *bar_k_free = bars, *bar_v_free = bars, *bar_k_full = bars, *bar_v_full = bars, *bar_dv_done = bars, *bar_dv_free = bars, *bar_dk_done = bars, *bar_dk_free = bars,
             *bar_g = bars, *bar_gfree = bars;
    auto begin = [] {};
    auto item_wait = [&](uint32_t) { ok &= warp_wait_relaxed(bars, 0); };
    auto item_read = [&](uint32_t i) { return items[i]; };
    auto item_at = [&](uint32_t i) { item_wait(i); Item it = item_read(i); if (!ok) it.n_sel = -1; return it; };
    auto warp_arrive = [](uint64_t*) {};
    me = warp & 3;
BODY
    left_ok = ok;
    std::lock_guard<std::mutex> l(m);
    ++gone;
    cv.notify_all();
}
// number of waits of the warp; -1: a barrier that not all four reach, -2: a warp that leaves without having learnt of the wait that gave up
extern "C" int run(int rows, int group, int failing, int at) {
    static __nv_bfloat16 data[512 * 2 * 64];
    static int32_t sel[512];
    P = Params{data, data, data, data, sel, nullptr, 512 * 128, 128, 64, 1, 512, 2, 64, 1, 1.f};
    arrived = gone = phase = 0; hung = false; fail_warp = failing; fail_at = at;
    for (int& w : waits) w = 0;
    bool ok[4];
    std::thread t[4];
    for (int w = 0; w < 4; ++w) t[w] = std::thread([=, &ok] { rows ? role<true>(4 + 4 * group + w, ok[w]) : role<false>(4 + 4 * group + w, ok[w]); });
    for (auto& x : t) x.join();
    if (hung) return -1;
    const bool gave_up = waits[failing] > at;
    for (bool o : ok) if (o == gave_up) return -2;
    return waits[failing];
}
"""


def test_warps_that_share_a_named_barrier_leave_together(tmp_path):
    """Nothing bounds a named barrier.  The warps that take results out in the many-tile backward share one: whichever wait of whichever warp gives up, all four learn of
    it and leave behind the same barrier.  The text of their branch, run on the host with every wait failing in turn."""
    body = next(text for fn, name, text in kernel_bodies() if name == "bwd_many_kernel")
    start = body.index("{", body.index("else if (warp < 12)")) + 1
    depth, end = 1, start
    while depth:
        depth += {"{": 1, "}": -1}.get(body[end], 0)
        end += 1
    text = re.sub(r"asm volatile[^\n]*", "", body[start:end - 1])
    assert "setmaxnreg" not in text and text.count("group_sync_and") >= 2
    (tmp_path / "role.cpp").write_text(HOST_WARPGROUP.replace("BODY", text))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-pthread", "-o", str(tmp_path / "role.so"), str(tmp_path / "role.cpp")])
    lib = C.CDLL(str(tmp_path / "role.so"))
    for rows in (0, 1):
        for group in (0, 1):
            for warp in range(4):
                waits = lib.run(rows, group, warp, 1 << 30)
                assert waits >= 3 + 6 + 3, "items, query tiles, finished items"
                got = [lib.run(rows, group, warp, at) for at in range(waits)]
                assert min(got) > 0, (rows, group, warp, got)


def test_shares_of_the_zero_rows_cover_every_row_once(tmp_path):
    """Where a CTA ends, the next one begins, however the compiler fuses products and sums: the shares of one build give the same rows in the other.  All rows are
    covered; an early CTA takes no fewer than a late one, and late ones keep their part of an even share."""
    (tmp_path / "rows.cpp").write_text('#include "attn_zero_rows.h"\nusing namespace vardrop;\n'
                                       'extern "C" void shares(int rows, int ctas, int early, float wanted, RowShares* s) { *s = row_shares(rows, ctas, early, wanted); }\n'
                                       'extern "C" void first(const RowShares* s, int* at) { for (int c = 0; c <= s->ctas; ++c) at[c] = first_row(*s, c); }\n')

    class Shares(C.Structure):
        _fields_ = [("rows", C.c_int), ("ctas", C.c_int), ("n_early", C.c_int), ("late", C.c_longlong), ("more", C.c_longlong)]

    libs = []
    fma = ["-mfma"] if " fma " in open("/proc/cpuinfo").read() else []
    for flags in (["-ffp-contract=off"], ["-ffp-contract=fast", *fma]):
        so = tmp_path / f"rows{len(libs)}.so"
        subprocess.check_call(["g++", "-std=c++17", "-O2", *flags, "-shared", "-fPIC", f"-I{ROOT}/paper_2501_14183_b200/csrc", "-o", str(so), str(tmp_path / "rows.cpp")])
        libs.append(C.CDLL(str(so)))
    for rows in (1, 2, 700, 1025, 8192 * 8, 5968 * 6, 2049 * 32, 32 * 65536, 2 ** 31 - 1):
        for ctas in (1, 2, 148, 1184, 1176, 5000):
            for early in {0, 1, ctas // 3, ctas - 1, ctas}:
                for wanted in (0.1, 3.7, 33.3, 1e4, 1e12):
                    s, at = Shares(), [(C.c_int * (ctas + 1))() for _ in libs]
                    libs[0].shares(rows, ctas, early, C.c_float(wanted), C.byref(s))
                    for lib, x in zip(libs, at):
                        lib.first(C.byref(s), x)
                    a, b = (np.ctypeslib.as_array(x) for x in at)
                    assert np.array_equal(a, b) and a[0] == 0 and a[-1] == rows and (np.diff(a) >= 0).all(), (rows, ctas, early, wanted)
                    assert s.more >= 0 and s.late * ctas >= rows * 1024 * (early / ctas if wanted > 1e3 else 0) * 0.99 - ctas, (rows, ctas, early, wanted)
                    assert a[-1] - a[-2] <= rows / ctas + 2 + ctas / 1024 + rows * 1e-6, (rows, ctas, early, wanted)


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
