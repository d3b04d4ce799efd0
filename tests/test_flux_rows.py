"""Where the corner fluxes of the persistent kernels go: every corner of an own vertex has a word of its own,
in bounds, and a vertex's words are its incidences in order, whatever its degree (host code)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I
from test_gpu_onchip import _fan
from test_gpu_vertex_degree import rect_hubs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_08241_gb300", "csrc")

PROGRAM = r"""
#include "sesw_internal.h"
using namespace sesw;
extern "C" long rows_check(int nv, int ne, const int32_t *tri, const double *xy, const double *pos, const double *depth,
                           const double *cor, int pv, int quads)
{
    sesw_mesh m{};
    m.nv = nv;
    m.ne = ne;
    m.tri = tri;
    m.xy = xy;
    m.pos = pos;
    m.depth = depth;
    m.coriolis = cor;
    HostMesh hm;
    std::string err;
    if (prepare_mesh(m, pv, hm, err) != 0 || build_halos(hm, err) != 0) return -1;
    int over = 0, verts = 0;
    for (int p = 0; p < hm.npatch; p++) {
        int o = 0;
        for (int v = hm.patch_v[p]; v < hm.patch_v[p + 1]; v++) o += overflow_quads(hm.vcsr_off[v + 1] - hm.vcsr_off[v]);
        over = std::max(over, o);
        verts = std::max(verts, hm.patch_v[p + 1] - hm.patch_v[p]);
    }
    long bad = 0;
    for (int p = 0; p < hm.npatch; p++) {
        const int v0 = hm.patch_v[p], nown = hm.patch_v[p + 1] - v0;
        const int s0 = hm.patch_slot[p], ns = hm.patch_slot[p + 1] - s0;
        // rows in arrays of quads, then the overflow quads (counted from the ninth flux on, whatever the rows
        // hold): which slot and corner writes each word
        const size_t o0 = 4 * (size_t)quads * verts;
        std::vector<int> who(o0 + 4 * (size_t)over, -1);
        for (int i = 0; i < ns; i++) {
            const ushort4 l = hm.slot_l[s0 + i];
            const uint2 f = hm.slot_f[s0 + i];
            const unsigned e[3] = {f.x & 0x1fffffu, (f.x >> 21) | ((f.y & 0x3ffu) << 11), (f.y >> 10) & 0x1fffffu};
            const unsigned lv[3] = {l.x, l.y, l.z};
            for (int c = 0; c < 3; c++) {
                const bool own = lv[c] < (unsigned)nown;
                if (own != (e[c] != 0x1fffffu)) bad++;
                if (!own) continue;
                size_t w = 4 * ((size_t)(e[c] >> 2) * verts + lv[c]) + (e[c] & 3);
                if (e[c] >= 4u * quads) w = o0 + 4 * (size_t)(hm.v_over[v0 + lv[c]] & 0xffffu) + (e[c] - 8);
                if (w >= who.size() || who[w] >= 0)
                    bad++;
                else
                    who[w] = 4 * i + c;
            }
        }
        // the vertex pass reads exactly the vertex's incidences in order
        for (int i = 0; i < nown; i++) {
            const int k0 = hm.vcsr_off[v0 + i], d = hm.vcsr_off[v0 + i + 1] - k0;
            const uint32_t o = hm.v_over[v0 + i];
            std::vector<int> seq;
            for (int k = 0; k < 4 * quads; k++) seq.push_back(who[4 * ((size_t)(k >> 2) * verts + i) + (k & 3)]);
            for (unsigned k = 4 * quads - 8; k < 4 * (o >> 16); k++)
                seq.push_back(who[o0 + 4 * (size_t)(o & 0xffffu) + k]);
            for (size_t k = 0; k < seq.size(); k++) bad += seq[k] != ((int)k < d ? (int)hm.vcsr[k0 + k] : -1);
            bad += (int)seq.size() < d;
        }
    }
    return bad;
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    cuda = "/usr/local/cuda/include"
    if not os.path.isdir(cuda):
        pytest.skip("no CUDA headers")
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    cuda, str(d / "rows.cpp"), os.path.join(CSRC, "mesh_prep.cpp"), "-o", str(d / "rows.so")], check=True)
    fn = ctypes.CDLL(str(d / "rows.so")).rows_check
    fn.restype = ctypes.c_long
    at = lambda a: a.ctypes.data_as(ctypes.c_void_p)   # noqa: E731
    return lambda m, pv: sum(fn(m.nv, m.ne, at(m.tri), at(m.xy), at(m.pos), at(m.depth), at(m.coriolis), pv, quads)
                             for quads in (2, 3, 4))


@pytest.mark.parametrize("degree", [7, 8, 9, 12, 13, 16, 17, 33, 100])
def test_hubs(check, degree):
    mesh = rect_hubs(101, 61, degree)
    for pv in (32, 45, 700):
        assert check(mesh, pv) == 0
    assert check(_fan(degree, 40), 32) == 0


def test_meshes_of_the_repository(check):
    assert check(I.channel_case(nx=61, ny=51).mesh, 100) == 0
    assert check(I.sphere_mesh(4), 50) == 0
