"""Which kernel takes a small mesh: the thread-block cluster under the automatic choice, the kernel with the
exchange through L2 where the caller names a residency or a form; sesw_info describes the one that runs."""
import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GRAPH, PERSISTENT = 1, 2
AUTO, REGISTERS, STREAM = 0, 1, 2


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2311_08241_gb300 import sesw

    sesw.load()
    return sesw


def _mesh(nx, ny):
    return I.tiny_jittered_case(nx=nx, ny=ny, seed=4).mesh


def _run(S, mesh, params, steps=(2,), mode=PERSISTENT, bps=0, form=AUTO):
    rng = np.random.default_rng(3)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        s.sesw_set_blocks_per_sm(bps)
        s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(params)
        s.sesw_set_state(eta, U)
        for n in steps:
            s.sesw_advance(n)
        out = s.sesw_get_state()
        assert s.sesw_status() == S.SESW_OK
        return out, s.sesw_get_info()


def _same(a, b, what):
    for x, y, name in zip(a, b, ("eta", "U", "<<U>>")):
        assert np.array_equal(x, y), f"{what}: {name} differs by {np.max(np.abs(x - y)):.3e}"


# vertices: too few patches for 8 blocks; 8 blocks; 16 blocks; too many slots for one per thread
@pytest.mark.parametrize("nx,ny,blocks", [(12, 14, 0), (17, 31, 16), (16, 20, 8), (60, 61, 16), (101, 51, 16),
                                          (95, 90, 0)])
def test_the_cluster_and_what_it_reports(S, nx, ny, blocks):
    mesh = _mesh(nx, ny)
    p = I.Params(tau=50.0, M=5)
    ref, _ = _run(S, mesh, p, mode=GRAPH)
    got, info = _run(S, mesh, p)
    assert info["mode"] == PERSISTENT and info["cluster_blocks"] == blocks, info
    if blocks:
        assert info["slots_per_thread"] == 1 and info["cached"] == 1 and info["launches"] == 1, info
        # one slot per thread: the blocks hold every slot
        assert info["block_threads"] * blocks >= info["nslot"] and info["block_threads"] <= 1024, info
    _same(ref, got, f"{blocks} blocks")


@pytest.mark.parametrize("bps,form", [(0, REGISTERS), (1, AUTO), (2, AUTO), (2, REGISTERS), (0, STREAM)])
def test_a_named_form_or_residency_is_taken(S, bps, form):
    mesh = _mesh(60, 61)
    p = I.Params(tau=50.0, M=5)
    ref, _ = _run(S, mesh, p, mode=GRAPH)
    got, info = _run(S, mesh, p, bps=bps, form=form)
    assert info["cluster_blocks"] == 0 and info["blocks_per_sm"] == (bps or 2), info
    assert (info["streamed"] != 0) == (form == STREAM), info
    _same(ref, got, f"form {form}, {bps} per SM")


def test_other_schemes_and_batches_do_not_report_it(S):
    mesh = _mesh(40, 37)
    _, info = _run(S, mesh, I.Params(tau=50.0, M=5, scheme=1))
    assert info["cluster_blocks"] == 0, info
    with S.Subcycle() as s:
        s.sesw_mesh_upload_batch([mesh, mesh])
        s.sesw_set_params_batch([I.Params(tau=50.0, M=5)] * 2)
        assert s.sesw_get_info()["cluster_blocks"] == 0


@pytest.mark.parametrize("steps", [1, 3])
@pytest.mark.parametrize("scheme,bps,form", [(0, 0, AUTO), (0, 2, AUTO), (0, 3, REGISTERS), (1, 0, AUTO), (1, 2, STREAM)])
def test_waits_give_up_and_the_context_goes_on(S, scheme, bps, form, steps):
    """Failure detection in the cluster, in the kernels with the exchange through L2 and in the last of several
    steps of one launch: one patch (one block of the cluster) publishes nothing in a launch's last step, the
    waits run out after about 10 ms each, and the same context and kernel then run normal steps, bitwise
    graph mode's."""
    import time

    mesh = _mesh(60, 61)
    p = I.Params(tau=40.0, M=5, scheme=scheme)
    rng = np.random.default_rng(3)
    eta, U = 0.3 * rng.standard_normal(mesh.nv), 5.0 * rng.standard_normal((mesh.ne, 2))
    ref, _ = _run(S, mesh, p, steps=[steps], mode=GRAPH)
    with S.Subcycle() as s:
        s.sesw_set_mode(PERSISTENT)
        s.sesw_set_blocks_per_sm(bps)
        s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        for _ in range(2):
            s.sesw_set_params(p, flags=S.SESW_FLAG_TEST_FORCE_TIMEOUT)
            assert (s.sesw_get_info()["cluster_blocks"] > 0) == (scheme == 0 and bps == 0)
            s.sesw_set_state(eta, U)
            t0 = time.perf_counter()
            s.sesw_advance(steps)
            assert s.sesw_status() == S.SESW_ETIMEOUT
            assert time.perf_counter() - t0 < 10.0
            s.sesw_set_params(p)
            s.sesw_set_state(eta, U)
            s.sesw_advance(steps)
            got = s.sesw_get_state()
            assert s.sesw_status() == S.SESW_OK
            _same(ref, got, "after a timeout")


@pytest.mark.parametrize("scheme,bps,form", [(0, 0, AUTO), (0, 2, AUTO), (0, 1, REGISTERS), (1, 2, AUTO), (1, 2, STREAM)])
@pytest.mark.parametrize("M,steps", [(200, 5), (512, 3), (513, 2), (7, 80)])
def test_steps_beyond_one_launch(S, scheme, bps, form, M, steps):
    """More substeps than one launch takes (512), in the cluster and in every kernel that takes several steps."""
    mesh = _mesh(41, 37)
    p = I.Params(tau=5.0 * M, M=M, scheme=scheme)
    ref, _ = _run(S, mesh, p, [1] * steps, GRAPH)
    got, info = _run(S, mesh, p, [steps], bps=bps, form=form)
    assert (info["cluster_blocks"] > 0) == (bps == 0 and scheme == 0), info
    _same(ref, got, f"M {M}, {steps} steps")
