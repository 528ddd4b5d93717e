"""The shared-memory image of the cluster-resident path holds every row that the bus step reads
without looking at a list's length (CPU: the layout function compiled into a small host program).

The bus step takes the first batch of a bus's lists unconditionally.  From an empty list at the end
of the bus order that is the generator row G, the line-end record 2 L, the phase row 2 L and the line
row 0, whether or not the network has generators or lines."""
import os
import subprocess

import pytest

from paper_2410_13055_gb300 import build as b

PROGRAM = r"""
#include "gx_internal.cuh"
#include <cstdio>
using namespace gx;
int main() {
    long bad = 0, n = 0;
    for (int N : {1, 3, 17}) for (int G : {0, 1, 9}) for (int L : {0, 1, 8}) for (int B : {0, 2, 5})
        for (int T : {1, 5, 24, 97}) for (int C : {1, 3, 16}) for (int V : {1, 4}) for (int adj : {0, 1}) {
            const int HS = crs_hours(T, C, V), nbo = (B + C - 1) / C, kw = T > 96 ? 2 : 1;
            if (HS * (C - 1) >= T) continue;
            const CrsOff o = crs_offsets(N, G, L, B, HS, C, T, B < nbo ? B : nbo, adj, 0, 128, V, kw);
            const size_t row = 4 * (size_t)HS;
            const bool ok = o.endr + 16 * (2 * (size_t)L + 1) <= o.liner &&  // the record past the last line end
                            o.xg + row * (G + 1) <= o.total &&               // the row past the last generator
                            o.dl + row <= o.q &&                             // line row 0
                            o.q + row * (2 * (size_t)L + 1) <= o.xb;         // the phase row past the last line end
            ++n;
            if (!ok && bad++ < 5) std::printf("N %d G %d L %d B %d T %d C %d V %d adj %d\n", N, G, L, B, T, C, V, adj);
        }
    std::printf("%ld of %ld outside\n", bad, n);
    return bad ? 1 : n > 500 ? 0 : 2;
}
"""


def test_unconditional_reads_of_the_bus_step_stay_in_the_image(tmp_path):
    nvcc = b._nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no CUDA compiler")
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, *b.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", b.CSRC, "-I",
                    os.path.join(os.path.dirname(b.HERE), "include"), str(src), "-o", str(exe)], check=True,
                   capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
