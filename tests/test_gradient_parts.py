"""The surrogate's weight gradients: how many rows one FP32 accumulator of the tensor cores adds up, and
where its partial sums go. An accumulator loses with every addition, so its run must not grow with the mesh."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_08241_gb300", "csrc")
MAX_ROWS = 2048

PROGRAM = r"""
#include <cstdio>
#include "sesw_internal.h"
int main()
{
    long n;
    while (scanf("%ld", &n) == 1) {
        const int N = (int)n, tiles = (N + sesw::kMsgTile - 1) / sesw::kMsgTile, ctas = sesw::bwd_layer_ctas(N);
        const int parts = sesw::bwd_layer_parts(N);
        std::vector<int> count(parts, 0);
        int bad = 0;
        for (int b = 0; b < ctas; b++)
            for (int t = b, done = 0; t < tiles; t += ctas, done++) {
                const int p = sesw::bwd_layer_part(ctas, b, done);
                if (p < 0 || p >= parts) bad++; else count[p]++;
            }
        int most = 0, least = 1 << 30;
        for (int c : count) { most = std::max(most, c); least = std::min(least, c); }
        printf("%d %d %d %d\n", bad, least, most * sesw::kMsgTile, ctas);
    }
}
"""


def test_every_partial_sum_is_written_and_short(tmp_path):
    src, exe = tmp_path / "parts.cpp", tmp_path / "parts"
    src.write_text(PROGRAM)
    cuda = next((d for d in ("/usr/local/cuda/include",) if os.path.isdir(d)), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    t = 128 * 304
    sizes = [1, 127, 128, 129, t - 1, t, t + 1, 16 * t - 128, 16 * t, 16 * t + 1, 16 * t + 129, 17 * t + 5, 32 * t,
             32 * t + 1, 910000, 3000000, 14680064, 200000000]
    out = subprocess.run([str(exe)], input="\n".join(map(str, sizes)), capture_output=True, text=True, check=True)
    for n, line in zip(sizes, out.stdout.splitlines()):
        bad, least, rows, ctas = map(int, line.split())
        assert bad == 0 and least >= 1, (n, line)      # no tile outside the buffer, no partial sum left unwritten
        assert rows <= MAX_ROWS, (n, line)
        assert 1 <= ctas <= 304, (n, line)


@pytest.mark.gpu
def test_gradient_error_does_not_grow_with_the_mesh():
    """3 M triangles: 9,868 rows per CTA. Against 64 bits the message layers' gradients stay within what 2048
    rows can lose: 256 additions of 16 rows (two per step) at half a unit of 24 bits each, and the 16 bits that
    the split of the incoming gradient carries."""
    import numpy as np
    import torch

    from perf import cases as C

    case, seed = {"kind": "train", "mesh": "rect", "nx": 1500, "ny": 1000}, 5
    exact = C.exact(case, seed)["grad"].ravel()
    torch.cuda.empty_cache()
    st = C.prepare(case, seed)
    got = torch.as_tensor(np.asarray(C.run(st)["grad"])).double().cuda().ravel()
    st["sim"].close()
    tol, o = 256 * 2.0 ** -24 + 2.0 ** -17, 0
    for i, (k, c) in enumerate(C._shapes()):
        n = k * c + c
        err = float((got[o:o + n] - exact[o:o + n]).norm() / exact[o:o + n].norm())
        if 2 <= i < 2 + 2 * C.LAYERS:
            assert err <= tol, (i, err, tol)
        o += n
