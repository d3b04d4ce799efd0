"""Graph mode's own choice of threads per block, bitwise against explicit block sizes: one partly filled
block, several rounds of the slot loop, one and several waves of blocks, turned neighbour frames."""
import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GRAPH = 1
MESHES = {
    "one-patch": lambda: I.tiny_jittered_case(nx=9, ny=8, seed=2),
    "small": lambda: I.tiny_jittered_case(nx=41, ny=33, seed=3),
    "waves": lambda: I.channel_case(nx=588, ny=340),
    "sphere": lambda: I.sphere_case(level=6),
}


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2311_08241_gb300 import sesw

    sesw.load()
    return sesw


def _run(S, mesh, params, threads):
    rng = np.random.default_rng(8)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    with S.Subcycle() as s:
        s.sesw_set_mode(GRAPH)
        if threads:
            s.sesw_set_block_threads(threads)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(params)
        s.sesw_set_forcing(1e-4 * rng.standard_normal((mesh.ne, 2)))
        s.sesw_set_state(eta, U)
        s.sesw_advance(2)
        assert s.sesw_status() == S.SESW_OK
        return s.sesw_get_state(), s.sesw_get_info()


@pytest.mark.parametrize("visc", [None, (1e-3, 1e-3)])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_block_size_does_not_change_results(S, name, visc):
    mesh = MESHES[name]().mesh
    p = I.Params(tau=9.0, M=3, visc=visc)
    ref, _ = _run(S, mesh, p, 256)
    for threads in (0, 64, 1024):
        got, info = _run(S, mesh, p, threads)
        assert info["block_threads"] == threads or (threads == 0 and info["block_threads"] % 32 == 0)
        for x, y, what in zip(ref, got, ("eta", "U", "<<U>>")):
            assert np.array_equal(x, y), f"{what} differs with {info['block_threads']} threads"
