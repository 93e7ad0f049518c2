"""The flux inlet's density (sums over the inlet's sites, the last block's total)
against the FP64 oracle at face sizes where it can go wrong: a single site, a
few, and more sites than the sums' grid has threads (GPU only). Compared are the
momentum populations, which the density sets at the face. (The components'
one-step bound is not for random phases at 46,000 sites: where the colour
gradient nearly cancels its direction is ill-conditioned, with and without
faces.) Tolerance: the one-step bound of 1e-6 max(|o|, t_q) and step."""
import numpy as np
import pytest

from lbm_cases import compare_state, pair, random_state, set_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 5), (3, 2, 4), (131, 127, 3)], ids=lambda s: "x".join(map(str, s)))
def test_flux_face_sizes(shape):
    nx, ny, nz = shape
    lab = np.zeros((nz, ny, nx), np.uint16)
    if nx > 3:
        lab[:, ::5, ::7] = 1
    n_in = int(np.count_nonzero(lab[0] == 0))
    dom, ref = pair(lab, None, (1, 1, 0), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95, force=(0.0, 0.0, 1e-5),
                    reservoir_z=3, rho_out=0.999, flux_in=0.003 * n_in)
    set_both(dom, ref, random_state(ref, seed=4, amp=0.02), 0)
    for k in range(1, 4):                       # the counter is back at zero for every launch
        dom.advance(1)
        ref.step(1)
        assert compare_state(dom, ref)[0] <= k * 1e-6
    dom.close()
