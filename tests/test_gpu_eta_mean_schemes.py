"""The step-mean elevation across a change of the scheme: it belongs to the SE scheme, and after a SESM
step it reads zero in every mode, never an earlier SE step's sum."""
import numpy as np
import pytest

from paper_2311_08241_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2], ids=["graph", "persistent"])
@pytest.mark.parametrize("steps", [1, 3])
@pytest.mark.parametrize("form", [0, 3])
def test_reads_zero_after_a_sesm_step(mode, steps, form):
    from paper_2311_08241_gb300 import sesw as S

    mesh = I.tiny_jittered_case(nx=61, ny=57, seed=4).mesh
    with S.Subcycle() as s:
        s.sesw_set_mode(mode)
        s.sesw_set_persistent_form(form)
        s.sesw_mesh_upload(mesh)
        s.sesw_set_params(I.Params(tau=50.0, M=5))
        s.sesw_set_eta_mean(True)
        s.sesw_set_state(np.full(mesh.nv, 0.25), np.zeros((mesh.ne, 2)))
        s.sesw_advance(steps)
        assert np.max(np.abs(s.sesw_get_eta_mean() - 0.25)) < 0.05
        s.sesw_set_params(I.Params(tau=50.0, M=5, scheme=1))
        s.sesw_advance(steps)
        assert not np.any(s.sesw_get_eta_mean())
        s.sesw_set_params(I.Params(tau=50.0, M=5))
        s.sesw_set_state(np.full(mesh.nv, 0.25), np.zeros((mesh.ne, 2)))
        s.sesw_advance(steps)
        assert np.max(np.abs(s.sesw_get_eta_mean() - 0.25)) < 0.05
