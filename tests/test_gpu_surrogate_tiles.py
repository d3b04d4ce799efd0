"""The surrogate's tile kernels at the edges of their tiles: rows that do not fill a tile of 128, fewer
rows than one tile, more tiles than thread blocks, vertices with many triangles (incidences that do
not fit shared memory), against the FP64 network of the oracle on the same bfloat16 values."""
import numpy as np
import pytest

from oracle import mpnn
from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2311_08241_gb300 import sesw

    sesw.load()
    return sesw


def _star(deg, copies):
    tri, P = [], []
    for c in range(copies):
        b = len(P)
        P.append((40e3 * c, 0.0))
        P += [(40e3 * c + 10e3 * np.cos(2 * np.pi * k / deg), 10e3 * np.sin(2 * np.pi * k / deg)) for k in range(deg)]
        tri += [(b, b + 1 + k, b + 1 + (k + 1) % deg) for k in range(deg)]
    P, tri = np.array(P), np.array(tri, dtype=np.int32)
    return I.Mesh("star", tri, np.ascontiguousarray(P[tri]), np.concatenate([P, np.zeros((len(P), 1))], 1),
                  np.linspace(1000.0, 3000.0, len(P)), np.full(len(tri), 1e-4))


def _mesh(name):
    """The mesh and the length scale of its element messages."""
    if name == "small":      # 7 x 6 vertices: less than one tile of rows of either kind
        return I.tiny_jittered_case(nx=7, ny=6, seed=2).mesh, 8e3
    if name == "star":       # one vertex with 2000 triangles: its tile's incidences exceed the shared list
        return _star(2000, 1), 30.0
    return I.channel_case(nx=190, ny=150).mesh, 8e3     # 442 tiles of element rows, 223 of vertex rows


@pytest.mark.parametrize("name", ["small", "star", "channel"])
def test_loss_and_gradient(S, name):
    mesh, length = _mesh(name)
    rng = np.random.default_rng(5)
    V, E = mesh.nv, mesh.ne
    f32 = lambda x: np.asarray(x, dtype=np.float32).astype(np.float64)   # noqa: E731
    eta, U, R = f32(0.3 * rng.standard_normal(V)), f32(3.0 * rng.standard_normal((E, 2))), \
        f32(1e-4 * rng.standard_normal((E, 2)))
    du, dm, de = f32(rng.standard_normal((E, 2))), f32(rng.standard_normal((E, 2))), f32(0.05 * rng.standard_normal(V))
    scales = [0.3, 3000.0, 3.0, 1e-4, 1e-4, length, 1.0, 0.05]
    with S.Subcycle() as s:
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(I.Params(tau=10.0, M=10), flags=S.SESW_FLAG_NO_STABILITY_CHECK)
        s.sesw_surrogate_init(1, seed=3)
        s.sesw_surrogate_scales(set=scales)
        w = (0.1 * rng.standard_normal(s.sesw_surrogate_nparam())).astype(np.float32)
        s.sesw_surrogate_weights(set=w)
        s.sesw_surrogate_set_sample(0, eta, U, R, du, dm, de)
        loss, grad = s.sesw_surrogate_gradient(0)
        again = s.sesw_surrogate_gradient(0)
        assert s.sesw_status() == S.SESW_OK
    assert again[0] == loss and np.array_equal(again[1], grad)
    sc = dict(zip(("eta", "H", "U", "R", "f", "L", "out_U", "out_eta"), scales))
    G = mpnn.Graph(mesh)
    xv, xe = mpnn.features(G, eta, U, R, sc)
    ref_loss, ref = mpnn.loss_and_grad(G, mpnn.quantise(w.astype(np.float64)), xv, xe,
                                       np.concatenate([du, dm], axis=1) / sc["out_U"], (de / sc["out_eta"])[:, None],
                                       sc, bf16_msgs=True)
    # The bounds of the small-mesh test of the same quantities: message inputs on a bfloat16
    # rounding boundary fall to either side (2^-8 apart), about 1e-4 of the gradient's scale.
    assert abs(loss - ref_loss) <= 1e-3 * abs(ref_loss)
    assert np.max(np.abs(grad - ref)) <= 1e-3 * np.max(np.abs(ref))
