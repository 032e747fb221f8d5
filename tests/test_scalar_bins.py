"""Which layers of scalar weights may use how many fine bins (csrc/idkm_scalar_bins.h): whole calls, on the CPU."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_07759_b200", "csrc")

PROGRAM = r"""
#include "idkm_scalar_bins.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {   // layers' sizes -> their bins, and the room the call reserves
  long long rows[64], total = 0;
  const int L = argc - 1;
  for (int l = 0; l < L; ++l) total += rows[l] = atoll(argv[l + 1]);
  for (int l = 0; l < L; ++l) {
    int larger = 0;
    for (int o = 0; o < L; ++o) larger += rows[o] > rows[l] || (rows[o] == rows[l] && o < l);
    std::printf("%d ", idkm::scalar_fine_bins(rows[l], larger, total));
  }
  std::printf("%d", idkm::scalar_fine_total(total, L));
}
"""
M = 1 << 20


def test_bins_of_whole_calls(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)])

    def call(*rows):
        out = [int(x) for x in subprocess.run([str(exe)] + [str(r) for r in rows], capture_output=True, text=True).stdout.split()]
        assert sum(out[:-1]) <= out[-1], rows
        return out[:-1]

    big, most, small = 32768, 40960, 16384
    assert call(4096) == [big] and call(8 * M) == [big] and call(10 * M - 1) == [big]
    assert call(10 * M) == [most] and call(44 * M) == [most] and call(44 * M - 9, 9) == [most, big]
    # places that do not fit in L2 with the weights, and several large layers: more bins are slower
    assert call(44 * M + 1) == [big] and call(64 * M) == [big] and call(44 * M, 1) == [big] * 2
    assert call(16 * M, 16 * M) == [big] * 2 and call(*[16 * M] * 4) == [big] * 4 and call(*[8 * M] * 8) == [big] * 8
    # the ninth largest and smaller ones, the largest first or last
    assert call(12 * M, *[1000] * 9) == [most] + [big] * 7 + [small] * 2
    assert call(*range(1, 10), 12 * M) == [small] * 2 + [big] * 7 + [most]
    assert call(*[4096] * 64) == [big] * 8 + [small] * 56
