"""The slots of an odd step (links.cuh) as 32-bit words, against the same in 64 bits, at
site counts up to the largest an image can have (no GPU: the functions compile for the
host)."""
import os
import subprocess

import host

SOURCE = r"""
#include <cstdio>
#include "links.cuh"
using namespace lbm;
int bad = 0;
char* const rows = reinterpret_cast<char*>(size_t{1} << 40);   // never read
void check(long long N) {
    const long long P = pitch_of(N);
    const long long ids[] = {0, 1, 31, N / 2, (1LL << 30) - 1, 1LL << 30, N - 2, N - 1};
    static_for<1, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        for (long long n : ids) {
            if (n < 0 || n >= N) continue;
            const long long alone = (opp(q) - q) * P + n;
            // through a word in memory, as the dense form keeps it
            const int word = static_cast<int>(slot_word<q>(false, -1, static_cast<int>(n), static_cast<int>(P)));
            bad += slot_at<q>(rows + q * P, static_cast<unsigned>(word)) - rows != q * P + alone;
            for (long long m : ids) {
                if (m < 0 || m >= N) continue;
                const int w = static_cast<int>(slot_word<q>(true, static_cast<int>(m), static_cast<int>(n), static_cast<int>(P)));
                bad += slot_at<q>(rows + q * P, static_cast<unsigned>(w)) - rows != q * P + m;
            }
        }
    });
}
int main() {
    for (long long N : {1LL, 31LL, 32LL, 33LL, 1000003LL, (1LL << 30) - 1, 1LL << 30, (1LL << 30) + 1, 1500000000LL,
                        (1LL << 31) - 4 * 1290 * 1290})
        check(N);
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_slots_at_any_size(tmp_path):
    src = tmp_path / "slots.cc"
    src.write_text(SOURCE)
    exe = tmp_path / "slots"
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-w", "-I", host.cuda_include(),
                    "-I", host.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
