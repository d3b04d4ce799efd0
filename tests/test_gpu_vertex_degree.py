"""Vertices of more than eight triangles on meshes of every size: the persistent SE kernel keeps the patch's
data on chip whatever the largest degree is, bitwise graph mode's results (one sequence of roundings in
every form)."""
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


def with_hubs(mesh, hubs, degree):
    """The mesh with vertices `hubs` (interior, no two of them within four edges of each other) raised to
    `degree` triangles: the edges opposite a hub are split, evenly one after another, together with the
    triangle behind them."""
    tri = mesh.tri
    order = np.argsort(tri.ravel(), kind="stable") // 3
    off = np.concatenate([[0], np.cumsum(np.bincount(tri.ravel(), minlength=mesh.nv))])
    at = lambda v: order[off[v]:off[v + 1]]   # noqa: E731
    drop, ntri, nxy, ncor, npos, ndep = [], [], [], [], [], []
    nv = mesh.nv

    def fan(t, k, chain, xs):
        """Triangle t, corner k against the chain of vertices that splits its opposite edge."""
        drop.append(t)
        x = mesh.xy[t]
        a, b = x[(k + 1) % 3], x[(k + 2) % 3]
        for i in range(len(chain) - 1):
            ntri.append((int(tri[t, k]), chain[i], chain[i + 1]))
            nxy.append((x[k], a + xs[i] * (b - a), a + xs[i + 1] * (b - a)))
            ncor.append(mesh.coriolis[t])

    for v in hubs:
        ts = at(v)
        need = degree - len(ts)
        for j, t in enumerate(ts):
            q = need // len(ts) + (j < need % len(ts))
            if q <= 0:
                continue
            k = int(np.nonzero(tri[t] == v)[0][0])
            a, b = int(tri[t, (k + 1) % 3]), int(tri[t, (k + 2) % 3])
            xs = np.linspace(0.0, 1.0, q + 2)
            chain = [a] + list(range(nv, nv + q)) + [b]
            nv += q
            for x in xs[1:-1]:
                npos.append(mesh.pos[a] + x * (mesh.pos[b] - mesh.pos[a]))
                ndep.append(mesh.depth[a] + x * (mesh.depth[b] - mesh.depth[a]))
            fan(t, k, chain, xs)
            for o in at(a):
                if o != t and b in tri[o]:
                    c = [i for i in range(3) if tri[o, i] not in (a, b)][0]
                    fan(o, c, chain[::-1], (1.0 - xs)[::-1])
    keep = np.ones(mesh.ne, dtype=bool)
    keep[drop] = False
    return I.Mesh(mesh.name + "_hubs",
                  np.ascontiguousarray(np.concatenate([tri[keep], np.array(ntri)]).astype(np.int32)),
                  np.ascontiguousarray(np.concatenate([mesh.xy[keep], np.array(nxy)])),
                  np.ascontiguousarray(np.concatenate([mesh.pos, np.array(npos)])),
                  np.concatenate([mesh.depth, np.array(ndep)]),
                  np.concatenate([mesh.coriolis[keep], np.array(ncor)]))


def rect_hubs(nx, ny, degree, every=12):
    """The rectangular basin with a hub at every `every`-th interior vertex in both directions."""
    mesh = I.basin_case(nx=nx, ny=ny, dx=10e3).mesh
    i, j = np.meshgrid(np.arange(5, nx - 5, every), np.arange(5, ny - 5, every))
    return with_hubs(mesh, (j * nx + i).ravel(), degree)


def _run(S, mesh, steps, mode, bps=0, form=0, scheme=0, extra=False):
    rng = np.random.default_rng(5)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        if mode == PERSISTENT:
            s.sesw_set_blocks_per_sm(bps)
            s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(I.Params(tau=6.0, M=3, scheme=scheme))
        if extra:
            s.sesw_set_freshwater(1e-6 * np.cos(np.arange(mesh.nv)))
            s.sesw_set_eta_mean(True)
        s.sesw_set_forcing(1e-4 * rng.standard_normal((mesh.ne, 2)))
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


@pytest.mark.parametrize("nx,ny,degree,bps,spt", [(901, 509, 9, 1, 7), (901, 509, 12, 1, 7), (901, 509, 17, 1, 7),
                                                  (588, 340, 9, 2, 3), (588, 340, 17, 2, 4), (250, 150, 33, 2, 1)])
def test_large_meshes_stay_on_chip(S, nx, ny, degree, bps, spt):
    """The automatic choice: a few vertices of high degree cost the others no shared memory, so that neither
    the streaming form nor one patch per SM is taken for them."""
    mesh = rect_hubs(nx, ny, degree)
    ref, _ = _run(S, mesh, [1, 1], GRAPH)
    got, info = _run(S, mesh, [2], PERSISTENT)
    assert info["streamed"] == 0 and info["blocks_per_sm"] == bps and info["slots_per_thread"] == spt, info
    _same(ref, got, f"degree {degree}")


@pytest.mark.parametrize("degree", [8, 9, 12, 13, 16, 17, 20, 41])
@pytest.mark.parametrize("bps", [0, 1, 4])
def test_overflow_quads_of_every_width(S, degree, bps):
    """Edges of the overflow quads, with the optional terms: in the cluster (bps 0, up to 16 triangles) and in the
    teams of the kernel with the exchange through L2."""
    mesh = rect_hubs(71, 43, degree, every=9)
    ref, _ = _run(S, mesh, [1, 1], GRAPH, extra=True)
    got, info = _run(S, mesh, [2], PERSISTENT, bps=bps, extra=True)
    assert (info["cluster_blocks"] > 0) == (bps == 0 and degree <= 16), info
    _same(ref, got, f"degree {degree}")


@pytest.mark.parametrize("degree", [8, 9, 13, 16, 17])
def test_sesm_teams(S, degree):
    """The SESM teams have the same rows up to 16 triangles; beyond them the mesh streams."""
    mesh = rect_hubs(201, 131, degree)
    ref, _ = _run(S, mesh, [1, 1], GRAPH, scheme=1)
    got, info = _run(S, mesh, [2], PERSISTENT, bps=2, form=2, scheme=1)
    assert info["streamed"] == 1, info
    _same(ref, got, f"degree {degree}")


def test_a_batch_with_one_such_basin(S):
    """Packs whose patches differ in their overflow: each basin as in its own upload."""
    meshes = [rect_hubs(101, 61, 8), rect_hubs(91, 71, 19), rect_hubs(61, 51, 9)]
    rng = np.random.default_rng(6)
    states = [(0.3 * rng.standard_normal(m.nv), 5.0 * rng.standard_normal((m.ne, 2))) for m in meshes]
    p = I.Params(tau=6.0, M=3)
    with S.Subcycle() as s:
        s.sesw_set_mode(PERSISTENT)
        s.sesw_mesh_upload_batch(meshes)
        s.sesw_set_params_batch([p] * 3)
        s.sesw_set_state(np.concatenate([e for e, _ in states]), np.concatenate([u for _, u in states]))
        s.sesw_advance(2)
        eta, U, _ = s.sesw_get_state()
    iv, ie = np.cumsum([m.nv for m in meshes])[:-1], np.cumsum([m.ne for m in meshes])[:-1]
    for m, (e, u), be, bu in zip(meshes, states, np.split(eta, iv), np.split(U, ie)):
        with S.Subcycle() as s:
            s.sesw_set_mode(GRAPH)
            s.sesw_mesh_upload(m)
            s.sesw_set_params(p)
            s.sesw_set_state(e, u)
            s.sesw_advance(1)
            s.sesw_advance(1)
            ge, gu, _ = s.sesw_get_state()
        assert np.array_equal(ge, be) and np.array_equal(gu, bu)
