"""CPU check of the base conversions' ranges: the host picks a target's scheme (bconv_target) by a proof
that its sums fit in 64 bits, and the rescale's lift adds more than 2^61 where the dropped limb has 61
bits. The function is compiled from the source as it stands; every scheme it picks is then run in exact
arithmetic at its extreme operands, over the prime sizes a context takes."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_00546_gb300", "csrc")

MAIN = r"""
// what bconv (bconv.cuh) computes with operands y and addend add, in 128 bits; false: a 64-bit step wrapped
static bool run(const BconvTarget& T, int ns, u64 y, u128 add, u64* out) {
    const u128 lim = (u128)1 << 64;
    bool ok = true;
    auto fold = [&](u128 v) {
        ok = ok && v < lim;
        const u32 vh = (u32)((u64)v >> 32), h = vh >> T.bsh;
        const u128 f = (u128)h * T.c + ((u64)(vh - (h << T.bsh)) << 32 | (u32)v);
        ok = ok && f < (u128)2 * T.q;
        return f;
    };
    const u32 xl = (u32)y, xh = (u32)(y >> 32);
    const int group = T.mode == 0 ? ns : 2;
    u128 sum = T.mode == 0 ? 0 : add;
    for (int i = 0; i < ns; i += group) {
        u128 a0 = T.mode == 0 ? add : 0, a1 = 0;
        for (int k = i; k < ns && k < i + group; ++k) {
            a1 += (u128)xl * T.hat[k].y + (u128)xh * T.hat[k].w;
            a0 += (u128)xl * T.hat[k].x + (u128)xh * T.hat[k].z;
            ok = ok && a1 < lim && a0 < lim;
        }
        const u128 r = a0 + (u128)(u32)a1 * T.mul + (u128)(u32)((u64)a1 >> 32) * T.c2;
        ok = ok && r < lim;
        if (T.mode == 0) sum = r;
        else sum += fold(r);
    }
    u128 f = fold(sum);
    *out = (u64)(f >= T.q ? f - T.q : f);
    return ok;
}

int main() {
    int picked[3] = {0, 0, 0}, bad = 0;
    for (int logn : {10, 13, 16})
        for (int b = 34; b <= 61; ++b) {
            std::vector<u64> pr, big;
            frh::gen_primes(logn, std::vector<int>(4, b), pr);
            frh::gen_primes(logn, {61}, big);
            for (u64 t : {pr.front(), pr.back()})
                for (int ns = 1; ns <= 8; ++ns)
                    for (u64 qmax : {t, big[0]}) {
                        const u128 add_max = std::max((u128)1 << 61, (u128)qmax + t);
                        for (u64 w : {t - 1, t / 2, (u64)1}) {
                            const std::vector<u64> hat(ns, w);
                            const BconvTarget T = bconv_target(t, hat, add_max);
                            ++picked[T.mode];
                            if (T.mode == 2) continue;
                            const u64 y = (u64)((1ull << 61) - 1);
                            for (u128 add : {(u128)0, (u128)qmax - 1 + t, add_max}) {
                                u64 got;
                                u128 ref = add % t;
                                for (int i = 0; i < ns; ++i) ref = (ref + (u128)(y % t) * w) % t;
                                if (!run(T, ns, y, add, &got) || got != (u64)ref) ++bad;
                            }
                        }
                    }
        }
    std::printf("%d %d %d %d\n", picked[0], picked[1], picked[2], bad);
    return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++") or not os.path.exists("/usr/local/cuda/include/vector_types.h"),
                    reason="needs g++ and the CUDA headers")
def test_schemes_hold_at_their_extremes(tmp_path):
    src = open(os.path.join(CSRC, "engine.cu")).read()
    parts = [re.search(r"^u64 inv_mod_2_64\(.*?^}", src, re.S | re.M).group(0),
             re.search(r"^u64 split30_host\(.*?}$", src, re.S | re.M).group(0),
             re.search(r"^BconvTarget bconv_target\(.*?^}", src, re.S | re.M).group(0)]
    head = ("#include <algorithm>\n#include <cstdint>\n#include <cstdio>\n#include <cstring>\n#include <vector>\n"
            "#include <vector_functions.h>\n#include \"fr_host.h\"\n"
            "typedef uint64_t u64;\ntypedef uint32_t u32;\ntypedef unsigned __int128 u128;\n")
    hdr = open(os.path.join(CSRC, "ckks_kernels.h")).read()
    head += re.search(r"^struct BconvTarget \{.*?^};", hdr, re.S | re.M).group(0) + "\n"
    (tmp_path / "t.cpp").write_text(head + "\n".join(parts) + MAIN)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", "-o", exe,
                    str(tmp_path / "t.cpp"), os.path.join(CSRC, "host_ring.cpp"), "-lpthread"], check=True)
    m0, m1, m2, bad = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert m0 > 0 and m1 > 0 and m2 > 0 and bad == 0
