"""The SESM kernels with several steps per launch, and the form for patches whose state but not static
data stays on chip, bitwise against graph mode (one sequence of roundings in every form)."""
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


def _run(S, mesh, params, steps, mode, bps=None, form=None, W=False):
    rng = np.random.default_rng(8)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    R = 1e-4 * rng.standard_normal((mesh.ne, 2))
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        if bps:
            s.sesw_set_blocks_per_sm(bps)
        if form is not None:
            s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(params)
        if W:
            s.sesw_set_freshwater(1e-6 * np.cos(np.arange(mesh.nv)))
        s.sesw_set_forcing(R)
        s.sesw_set_state(eta, U)
        for n in steps:
            s.sesw_advance(n)
        out = s.sesw_get_state()
        assert s.sesw_status() == S.SESW_OK
        return out, s.sesw_get_info()


def _same(a, b, what):
    for x, y, name in zip(a, b, ("eta", "U", "<<U>>")):
        assert np.array_equal(x, y), f"{what}: {name} differs by {np.max(np.abs(x - y)):.3e}"


@pytest.mark.parametrize("M,parts", [(1, [3]), (2, [1, 2]), (9, [4]), (200, [5])])
@pytest.mark.parametrize("form", [0, 2])
def test_several_steps_per_launch(S, M, parts, form):
    mesh = I.tiny_jittered_case(nx=61, ny=57, seed=4).mesh
    p = I.Params(tau=10.0 * M, M=M, scheme=1)
    ref, _ = _run(S, mesh, p, [1] * sum(parts), GRAPH, W=True)
    _same(ref, _run(S, mesh, p, [1] * sum(parts), PERSISTENT, form=form, W=True)[0], "single steps")
    _same(ref, _run(S, mesh, p, parts, PERSISTENT, form=form, W=True)[0], f"steps {parts}")


@pytest.mark.parametrize("nx,ny,bps,spt", [(588, 340, 1, 4), (320, 310, 4, 4), (560, 560, 1, 5), (620, 620, 1, 6),
                                           (640, 620, 2, 6), (690, 690, 1, 7)])
def test_slots_per_thread(S, nx, ny, bps, spt):
    mesh = I.channel_case(nx=nx, ny=ny).mesh
    p = I.Params(tau=15.0, M=3, scheme=1)
    ref, _ = _run(S, mesh, p, [2], GRAPH)
    got, info = _run(S, mesh, p, [2], PERSISTENT, bps=bps, form=2)
    assert info["slots_per_thread"] == spt and info["streamed"] == 1, info
    _same(ref, got, f"{spt} slots per thread")
