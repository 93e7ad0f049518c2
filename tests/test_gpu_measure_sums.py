"""The analysis' sums (warp sums of compensated pairs, the last block's total)
against the FP64 oracle at site counts where they can go wrong: one site, part of a
warp, a full block and one site more, and more sites than the smallest grid has
threads (GPU only). Tolerance: the fp32 sums inside a site are all that differs, at
most 19 roundings of 2^-24, 1.2e-6 of the sum of magnitudes."""
import numpy as np
import pytest

from lbm_cases import pair, random_state, set_both

pytestmark = pytest.mark.gpu

BOUND = 19 * 2.0 ** -24


@pytest.mark.parametrize("parity", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 1), (7, 3, 1), (16, 16, 1), (257, 1, 1), (61, 59, 53)],
                         ids=lambda s: "x".join(map(str, s)))
def test_measure_sums(shape, parity):
    nx, ny, nz = shape
    dom, ref = pair(np.zeros((nz, ny, nx), np.uint16), None, (1, 1, 1), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95)
    set_both(dom, ref, random_state(ref, seed=3), parity)
    o = ref.measure()
    first = dom.measure()
    for k in ("mass_a", "mass_b", "mass_total"):
        assert abs(first[k] - o[k]) <= BOUND * abs(o[k]), k
    # magnitudes of a site's momentum: the populations leaving along an axis, about 1/3
    for i, k in enumerate(("flux_x", "flux_y", "flux_z")):
        assert abs(first["flux"][i] - o[k]) <= BOUND, k
    for _ in range(2):                          # the counter of finished blocks is back at zero
        assert dom.measure() == first
    dom.close()
