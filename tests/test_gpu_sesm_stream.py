"""The streaming SESM kernel with the slots' corner indices in shared memory (k_persistent_sesm_stream), which runs
where the teams' kernel does not: patches beyond 7 slots per thread, and meshes with a vertex of more than 16
triangles. Bitwise against graph mode. (Teams report 4 to 7 slots per thread, this kernel its rounds.)"""
import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I
from test_gpu_vertex_degree import rect_hubs

pytestmark = pytest.mark.gpu
GRAPH, PERSISTENT = 1, 2


def _run(mesh, params, steps, mode, bps=0, form=0, W=False):
    from paper_2311_08241_gb300 import sesw as S

    rng = np.random.default_rng(8)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        if mode == PERSISTENT:
            s.sesw_set_blocks_per_sm(bps)
            s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(params)
        if W:
            s.sesw_set_freshwater(1e-6 * np.cos(np.arange(mesh.nv)))
        s.sesw_set_forcing(1e-4 * rng.standard_normal((mesh.ne, 2)))
        s.sesw_set_state(eta, U)
        for n in steps:
            s.sesw_advance(n)
        out = s.sesw_get_state()
        assert s.sesw_status() == S.SESW_OK
        return out, s.sesw_get_info()


def _same(a, b):
    for x, y, name in zip(a, b, ("eta", "U", "<<U>>")):
        assert np.array_equal(x, y), f"{name} differs by {np.max(np.abs(x - y)):.3e}"


@pytest.mark.parametrize("M,steps", [(1, [3]), (2, [1, 2]), (9, [2])])
@pytest.mark.parametrize("bps,nonlinear", [(1, 1), (2, 0), (4, 1)])
def test_small_patches(M, steps, bps, nonlinear):
    mesh = rect_hubs(131, 97, 17)
    p = I.Params(tau=2.0 * M, M=M, scheme=1, nonlinear_h=nonlinear)
    ref, _ = _run(mesh, p, [1] * sum(steps), GRAPH, W=True)
    got, info = _run(mesh, p, steps, PERSISTENT, bps=bps, form=2, W=True)
    assert info["streamed"] == 1 and info["slots_per_thread"] < 4, info
    _same(ref, got)


def test_patches_beyond_the_teams():
    mesh = I.basin_case(nx=740, ny=702, dx=10e3).mesh
    p = I.Params(tau=20.0, M=2, scheme=1)
    ref, _ = _run(mesh, p, [1, 1], GRAPH)
    got, info = _run(mesh, p, [2], PERSISTENT, bps=1)
    assert info["streamed"] == 1 and info["slots_per_thread"] == 8, info
    _same(ref, got)
