"""The persistent SE kernel's on-chip data (tensor memory, flux rows of the vertices, teams) at the
edges of its layouts. Every form of the SE scheme rounds in one order, so each run must be bitwise
the graph mode's."""
import dataclasses

import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GRAPH, PERSISTENT = 1, 2


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2311_08241_gb300 import sesw

    sesw.load()
    return sesw


def _state(mesh, seed=3):
    rng = np.random.default_rng(seed)
    return 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2)), \
        1e-4 * rng.standard_normal((mesh.ne, 2))


def _run(S, mesh, params, steps, mode, bps=None, form=None, extra=False):
    eta, U, R = _state(mesh)
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        if bps:
            s.sesw_set_blocks_per_sm(bps)
        if form is not None:
            s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(params)
        if extra:
            s.sesw_set_freshwater(1e-6 * np.cos(np.arange(mesh.nv)))
            s.sesw_set_eta_mean(True)
        s.sesw_set_forcing(R)
        s.sesw_set_state(eta, U)
        for n in steps:
            s.sesw_advance(n)
        out = list(s.sesw_get_state())
        if extra:
            out.append(s.sesw_get_eta_mean())
        assert s.sesw_status() == S.SESW_OK
        return out, s.sesw_get_info()


def _same(a, b, what):
    for x, y, name in zip(a, b, ("eta", "U", "<<U>>", "eta_bar")):
        assert np.array_equal(x, y), f"{what}: {name} differs by {np.max(np.abs(x - y)):.3e}"


def _fan(deg, copies):
    """`copies` separate fans of `deg` triangles around one vertex each (closed rings)."""
    tri, P = [], []
    for c in range(copies):
        b = len(P)
        P.append((40e3 * c, 0.0))
        for k in range(deg):
            a = 2.0 * np.pi * k / deg
            P.append((40e3 * c + 10e3 * np.cos(a), 10e3 * np.sin(a)))
        tri += [(b, b + 1 + k, b + 1 + (k + 1) % deg) for k in range(deg)]
    P, tri = np.array(P), np.array(tri, dtype=np.int32)
    return I.Mesh("fan", tri, np.ascontiguousarray(P[tri]), np.concatenate([P, np.zeros((len(P), 1))], 1),
                  np.full(len(P), 3000.0), np.full(len(tri), 1e-4))


@pytest.mark.parametrize("deg", [3, 4, 5, 8, 9, 12, 13, 16, 17])
def test_vertex_rows_of_every_width(S, deg):
    """Rows of 8, 12 and 16 fluxes, and vertices with more (data from L2)."""
    mesh = _fan(deg, 40)
    p = I.Params(tau=20.0, M=5)
    ref, _ = _run(S, mesh, p, [2], GRAPH)
    got, info = _run(S, mesh, p, [2], PERSISTENT)
    assert info["cached"] == (1 if deg <= 16 else 0), info
    _same(ref, got, f"degree {deg}")


@pytest.mark.parametrize("M,parts", [(1, [3]), (1, [1, 2]), (3, [2]), (7, [5]), (7, [1, 4]), (200, [5])])
@pytest.mark.parametrize("extra", [False, True])
def test_several_steps_per_launch(S, M, parts, extra):
    """One launch of n steps against single steps, with the optional terms too; (200, [5]) needs more
    than one launch."""
    mesh = I.tiny_jittered_case(nx=41, ny=37, seed=4).mesh
    p = I.Params(tau=10.0 * M, M=M)
    ref, _ = _run(S, mesh, p, [1] * sum(parts), GRAPH, extra=extra)
    one, _ = _run(S, mesh, p, [1] * sum(parts), PERSISTENT, extra=extra)
    got, _ = _run(S, mesh, p, parts, PERSISTENT, extra=extra)
    _same(ref, one, "single steps")
    _same(ref, got, f"steps {parts}")


@pytest.mark.parametrize("bps", [1, 2, 3, 4])
def test_teams_with_more_halo_vertices_than_threads(S, bps):
    """Vertices in random order (no positions): a patch's halo is several times its own vertices."""
    case = I.channel_case(nx=211, ny=191)
    rng = np.random.default_rng(1)
    perm = rng.permutation(case.mesh.nv)
    m = case.mesh
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    mesh = dataclasses.replace(m, tri=inv[m.tri].astype(np.int32), pos=None, depth=m.depth[perm])
    mesh.__class__ = _NoPos
    p = I.Params(tau=60.0, M=3)
    ref, _ = _run(S, mesh, p, [2], GRAPH)
    got, info = _run(S, mesh, p, [2], PERSISTENT, bps=bps)
    assert info["mode"] == PERSISTENT
    _same(ref, got, f"{bps} teams per SM")


class _NoPos(I.Mesh):
    @property
    def nv(self):
        return int(self.depth.shape[0])


@pytest.mark.parametrize("nx,ny,bps,spt", [(300, 300, 1, 2), (500, 480, 1, 4), (600, 560, 1, 5), (640, 620, 1, 6),
                                           (640, 620, 2, 6)])
def test_slots_per_thread(S, nx, ny, bps, spt):
    """Each split of the slots' data between tensor memory, shared memory and L2 (3 and 7 slots per
    thread are covered by the channel and the level-8 sphere)."""
    case = I.channel_case(nx=nx, ny=ny)
    p = I.Params(tau=20.0, M=3)
    ref, _ = _run(S, case.mesh, p, [2], GRAPH)
    got, info = _run(S, case.mesh, p, [2], PERSISTENT, bps=bps, form=1)
    assert info["slots_per_thread"] == spt and info["streamed"] == 0, info
    _same(ref, got, f"{spt} slots per thread")


@pytest.mark.parametrize("nx,ny", [(16, 16), (17, 31), (23, 23), (40, 37), (60, 61), (66, 64)])
@pytest.mark.parametrize("M,parts", [(1, [1]), (1, [2]), (2, [1, 3]), (9, [2])])
def test_small_meshes_in_one_cluster(S, nx, ny, M, parts):
    """The cluster of 8 or 16 blocks that takes small meshes (up to one slot per thread), from too few
    patches for it to too many slots, with every optional term, against graph mode and against the
    kernel that exchanges through L2 (an explicit residency)."""
    mesh = I.tiny_jittered_case(nx=nx, ny=ny, seed=4).mesh
    p = I.Params(tau=10.0 * M, M=M)
    for extra in (False, True):
        ref, _ = _run(S, mesh, p, [1] * sum(parts), GRAPH, extra=extra)
        got, info = _run(S, mesh, p, parts, PERSISTENT, extra=extra)
        assert info["mode"] == PERSISTENT
        _same(ref, got, "cluster")
        _same(ref, _run(S, mesh, p, parts, PERSISTENT, bps=2, extra=extra)[0], "through L2")


def test_small_mesh_of_separate_parts(S):
    """Disconnected fans: blocks of a cluster that read nothing from the others."""
    mesh = _fan(6, 120)
    p = I.Params(tau=20.0, M=5)
    ref, _ = _run(S, mesh, p, [2], GRAPH)
    _same(ref, _run(S, mesh, p, [2], PERSISTENT)[0], "fans")
