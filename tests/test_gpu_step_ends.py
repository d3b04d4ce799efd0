"""The end of a step inside a launch of several, where the compensated sums start again: with their low
parts in shared memory (6 to 8 slots per thread) every element's mean must be the single steps', bit
for bit."""
import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GRAPH, PERSISTENT = 1, 2


class _NoPos(I.Mesh):
    @property
    def nv(self):
        return int(self.depth.shape[0])


def _mesh(nx, ny, shuffled):
    m = I.channel_case(nx=nx, ny=ny).mesh
    if not shuffled:
        return m
    # vertices in random order: a patch of few vertices holds many triangles
    perm = np.random.default_rng(1).permutation(m.nv)
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    return _NoPos(m.name, np.ascontiguousarray(inv[m.tri].astype(np.int32)), m.xy, None,
                  np.ascontiguousarray(m.depth[perm]), m.coriolis)


def _run(S, mesh, mode, steps):
    rng = np.random.default_rng(3)
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        if mode == PERSISTENT:
            s.sesw_set_blocks_per_sm(1)
            s.sesw_set_persistent_form(1)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(I.Params(tau=12.0, M=3))
        s.sesw_set_state(0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2)))
        for n in steps:
            s.sesw_advance(n)
        return s.sesw_get_state(), s.sesw_get_info()


@pytest.mark.parametrize("nx,ny,shuffled,spt", [(640, 620, False, 6), (690, 690, False, 7), (440, 430, True, 8)])
def test_sums_start_again(nx, ny, shuffled, spt):
    from paper_2311_08241_gb300 import sesw as S

    mesh = _mesh(nx, ny, shuffled)
    ref, _ = _run(S, mesh, GRAPH, [1] * 4)
    got, info = _run(S, mesh, PERSISTENT, [4])
    assert info["slots_per_thread"] == spt and info["cached"] == 2, info
    for a, b, name in zip(ref, got, ("eta", "U", "<<U>>")):
        assert np.array_equal(a, b), name
