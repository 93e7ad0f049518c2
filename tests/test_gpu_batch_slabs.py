"""The batch's reservoir reset (one launch for up to 32 jobs) against the same jobs
advanced alone, at job counts around the table's size, with slabs of part of a tile
and of several, jobs without slabs between them, and a job with pressure faces, whose
population form the whole batch then takes (GPU only). Tolerance: the one of batched
against single-domain runs, 1e-5 per distribution."""
import numpy as np
import pytest

from lbm_cases import T19, W7

pytestmark = pytest.mark.gpu


def _job(i, precision, faces):
    import paper_2007_12266_gb300 as lbm
    nx, ny, nz = (3 + i % 5, 4, 9) if i % 8 else (23, 19, 10)
    lab = np.zeros((nz, ny, nx), np.uint16)
    lab[::2, 1, 1] = 1
    slabs = i % 3 != 1                           # reservoir slabs, or a periodic z axis
    kw = dict(reservoir_z=2 if faces else 1, rho_in=1.001, rho_out=0.999) if slabs or faces else {}
    d = lbm.Domain(lab, (0.4 * lab).astype(np.float32), periodic=(1, 1, 0 if kw else 1), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95,
                   force=(0.0, 0.0, 1e-5), precision=precision, **kw)
    d.init_fluids(np.where(np.arange(nz)[:, None, None] < 4, 0.8, -0.9) * np.ones((nz, ny, nx)))
    return d


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("slab_jobs,faces", [(1, False), (32, False), (33, False), (33, True)])
def test_batch_slabs(slab_jobs, faces, precision):
    import paper_2007_12266_gb300 as lbm
    n = (slab_jobs * 3 + 1) // 2                 # two of three jobs have slabs
    kinds = [False] * n + ([True] if faces else [])
    alone = [_job(i, precision, k) for i, k in enumerate(kinds)]
    batched = [_job(i, precision, k) for i, k in enumerate(kinds)]
    b = lbm.Batch()
    for d in batched:
        b.add(d)
    b.advance(8)
    for d in alone:
        if faces:
            d.set_step_form("populations")        # the batch's form
        d.advance(8)
    for da, db in zip(alone, batched):
        for which, floor in (("f", T19), ("a", W7), ("b", W7)):
            x, y = da.distributions(which).astype(np.float64), db.distributions(which).astype(np.float64)
            assert (np.abs(x - y) / np.maximum(np.abs(x), floor[:, None])).max() <= 1e-5
    b.close()
    for d in alone + batched:
        d.close()
