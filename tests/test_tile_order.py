"""The persistent contraction's tile order (``tcp_pick``), compiled from the kernel source: every
tile is taken exactly once, a CTA that runs past the end of the table is done, and the pairs of
rounds balance a table sorted longest first."""
import pathlib
import re
import subprocess

SRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2408_04875_gb300" / "csrc" / "tc_gemm.cu"

HARNESS = r"""
#include <cstdio>
#define __device__
#define __forceinline__ inline
struct Dim { unsigned x; } gridDim, blockIdx;
%s
int main()
{
    const int grids[] = {1, 2, 3, 7, 151, 152}, sizes[] = {0, 1, 2, 3, 151, 152, 153, 179, 303, 304, 305, 5000};
    long bad = 0;
    for (int g : grids)
        for (int n : sizes) {
            static int seen[5000];
            for (int i = 0; i < n; ++i) seen[i] = 0;
            gridDim.x = (unsigned)g;
            for (int b = 0; b < g; ++b) {
                blockIdx.x = (unsigned)b;
                int rd = 0, t;
                for (; (t = tcp_pick(rd)) < n; ++rd) {
                    if (t < 0) return 2;
                    seen[t] += 1;
                }
                for (int later = rd; later < rd + 4; ++later) bad += tcp_pick(later) < n;
                bad += tcp_pick(0) + tcp_pick(1) != 2 * g - 1;   // as many places from the front as from the back
            }
            for (int i = 0; i < n; ++i) bad += seen[i] != 1;
        }
    std::printf("%%ld\n", bad);
    return 0;
}
"""


def test_every_tile_once(tmp_path):
    body = re.search(r"__device__ __forceinline__ int tcp_pick\(int rd\)\n\{.*?\n\}\n", SRC.read_text(), re.S).group(0)
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(HARNESS % body)
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
