"""Host side of the kernel dispatch: launches that no kernel can take are refused before
anything is launched (no GPU is needed or used)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INVALID_VALUE = 1


def test_generic_kernel_is_refused_for_launches_with_bins(tmp_path):
    """A launch that clears or fills the bins of an exact sum, or has an extra step, and that the
    tuned kernels do not take (here: no recurrence coefficients, an odd Ls, an untuned even Ls)
    gives cudaErrorInvalidValue: the generic kernel would leave the bins uncleared."""
    cxx, cuda = shutil.which("g++"), "/usr/local/cuda"
    if cxx is None or not os.path.exists(cuda + "/include/cuda_runtime.h"):
        pytest.skip("no C++ compiler or no CUDA headers")
    from paper_1501_04950_gb300.build import build
    lib = build()
    src = tmp_path / "refuse.cpp"
    src.write_text(r"""
#include <cstdio>
#include "dwf_internal.cuh"
using namespace dwf;
int main() {
  bin_t* word = reinterpret_cast<bin_t*>(256);  // never read
  for (int Ls : {8, 7, 14})
    for (int prec : {P64, P32, P16, PB16})
      for (int k = 0; k < 4; k++) {
        Geom g{{4, 4, 4, 4}, 2, 128, Ls, 128 * Ls, 1};
        Reduce red{};
        HopLaunch L{};
        L.prec = prec;
        L.nrhs = 1;
        L.loc = LOC_ID;
        L.c_loc = 1.0;
        L.post = word;
        L.post_prog = 2;  // I^-1
        if (k < 2) L.zero[k] = word;
        if (k == 2) { red.bins = word; L.red = &red; }
        if (k == 3) L.extra = 1;
        std::printf("%d\n", (int)launch_hop(g, L, nullptr));
      }
}
""")
    exe = tmp_path / "refuse"
    subprocess.run([cxx, "-std=c++17", "-I", cuda + "/include",
                    "-I", os.path.join(ROOT, "paper_1501_04950_gb300", "csrc"), str(src), lib,
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert len(out) == 48
    assert set(out) == {str(CUDA_INVALID_VALUE)}
