"""The collision's two FP32 block sizes on either side of the site count where the
dispatch changes, against the same domain in a batch, whose blocks are of another size
(GPU only). Tolerance: the one of batched against single-domain runs, 1e-5."""
import numpy as np
import pytest

from lbm_cases import T19, W7

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["auto", "populations"])
@pytest.mark.parametrize("solids", [0, 1])
def test_block_sizes(solids, form):
    import paper_2007_12266_gb300 as lbm
    lab = np.zeros((64, 128, 128), np.uint16)    # 2^20 sites
    lab.ravel()[5:5 + solids] = 1
    phi0 = np.random.default_rng(1).uniform(-0.9, 0.9, lab.shape)
    doms = []
    for _ in range(2):
        d = lbm.Domain(lab, None, periodic=(1, 1, 1), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95,
                       force=(0.0, 0.0, 1e-5))
        d.set_step_form(form)
        d.init_fluids(phi0)
        doms.append(d)
    assert doms[0].n_sites == (1 << 20) - solids
    b = lbm.Batch()
    b.add(doms[1])
    doms[0].advance(4)
    b.advance(4)
    for which, floor in (("f", T19), ("a", W7), ("b", W7)):
        x, y = (d.distributions(which).astype(np.float64) for d in doms)
        assert (np.abs(x - y) / np.maximum(np.abs(x), floor[:, None])).max() <= 1e-5
    b.close()
    for d in doms:
        d.close()
