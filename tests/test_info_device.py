"""sesw_get_info of a context on one device while another is current: what it asks of the CUDA runtime is
asked on the context's device, and the caller's device is current again afterwards (host code against a
fake runtime with two devices)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_08241_gb300", "csrc")

PROGRAM = r"""
#include "sesw_api.cpp"
static int current = 0, asked_on = -1;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
extern "C" cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
namespace sesw {
int substep_threads(const DevMesh &, bool, bool) { asked_on = current; return 320; }
}
int main()
{
    sesw_ctx c;
    c.device = 1;
    c.mode = SESW_MODE_GRAPH;
    c.have_mesh = c.have_params = true;
    c.params.M = 3;
    sesw_info info;
    const int rc = sesw_get_info(&c, &info);
    printf("%d %d %d %d\n", rc, info.block_threads, asked_on, current);
}
"""


def test_asks_on_the_contexts_device(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not os.path.isdir(cuda):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "info.cpp", tmp_path / "info"
    src.write_text(PROGRAM)
    # only the three functions above run; the library's other symbols stay unresolved
    subprocess.run(["g++", "-std=c++17", "-no-pie", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda, str(src),
                    "-o", str(exe), "-Wl,--unresolved-symbols=ignore-all", "-pthread"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["0", "320", "1", "0"], out
