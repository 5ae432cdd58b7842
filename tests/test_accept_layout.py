"""The scratch of the accept call: what its passes keep fits at every size, in the bytes that callers have been asked for all along, and
no size is left that only the one-cluster resample could take.  The host header, compiled with the host compiler."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "accept_layout.cuh"
#include <cstdio>
#include <initializer_list>

int main() {
    int wrong = 0;
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    for (int times : {1, 4})
        for (int rows : {1, 2, 3, 7, 16, 31, 32, 33, 64, 128, 300, 4096})
            for (int k : {0, 1, 16})
                for (int V = 1; V <= 300000; V += V < 20000 ? 1 : 509) {
                    const csd::AcceptLayout L = csd::accept_layout(rows, k, V, times);
                    const size_t n = (V + 512 * times - 1) / (512 * times), r = rows;
                    const size_t asked = up(r * (2 * k + 1) * ((V + 8191) / 8192) * 16) + up(r * 48) + up(r * n * 16) + up(r * n * 8) + up(r * 16) + up(r * 8);
                    const bool fits = L.info_off >= r * (2 * k + 1) * L.nchunk_a * 16 && L.sums_off >= L.info_off + r * 48 &&
                                      L.lists_off >= L.sums_off + r * L.chunks * 32 && L.ticket_off >= L.lists_off + r * L.chunks * 12 &&
                                      L.total >= L.ticket_off + r * 4;
                    const bool covers = (long long)L.chunks * L.sets * 512 >= V && (long long)(L.chunks - 1) * L.sets * 512 < V;
                    const bool aligned = L.info_off % 16 == 0 && L.sums_off % 16 == 0 && L.lists_off % 4 == 0 && L.ticket_off % 4 == 0;
                    if (L.total != asked || !fits || !covers || !aligned) ++wrong;
                }
    std::printf("%d\n", wrong);
    return wrong != 0;
}
"""


def test_what_the_passes_keep_fits(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2312_11462_b200", "csrc"), "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True, timeout=60).stdout == "0\n"
