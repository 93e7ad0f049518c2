"""The component populations that a pressure or flux face sets, against the FP64 oracle
at faces of a few sites, beside the momentum populations (GPU only). Tolerance: the
one-step bound of 1e-6 max(|o|, t_q or w_q) and step."""
import numpy as np
import pytest

from lbm_cases import compare_state, pair, random_state, set_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [0, 1])
@pytest.mark.parametrize("face", [dict(reservoir_z=2, rho_in=1.003, rho_out=0.998), dict(reservoir_z=3, rho_out=0.999)],
                         ids=["pressure", "flux"])
@pytest.mark.parametrize("shape", [(1, 1, 5), (3, 2, 4), (7, 6, 4)], ids=lambda s: "x".join(map(str, s)))
def test_components_at_small_faces(shape, face, start):
    nx, ny, nz = shape
    lab = np.zeros((nz, ny, nx), np.uint16)
    if face["reservoir_z"] == 3:
        face = dict(face, flux_in=0.003 * nx * ny)
    dom, ref = pair(lab, None, (1, 1, 0), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95, force=(0.0, 0.0, 1e-5), **face)
    set_both(dom, ref, random_state(ref, seed=4, amp=0.02), start)
    for k in range(1, 4):
        dom.advance(1)
        ref.step(1)
        assert max(compare_state(dom, ref)) <= k * 1e-6
    dom.close()
