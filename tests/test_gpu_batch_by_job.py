"""Batches of large jobs run job by job on several streams with the default launch
shape: the same result, bit for bit, as one launch per pass over all jobs, on either
side of the mean job size where the dispatch changes, with more jobs than streams, a
reservoir job and a job with a periodic x axis (GPU only). A served job's result must
not depend on which of the two ran it, hence no tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EDGES = [(40, 40, 36), (64, 32, 32), (41, 41, 41), (40, 64, 28), (33, 64, 31)]


def _domains(precision, grow):
    import paper_2007_12266_gb300 as lbm
    doms = []
    for i, (nx, ny, nz) in enumerate(EDGES):
        lab = np.zeros((nz + grow, ny, nx), np.uint16)
        lab[::5, ::6, ::7] = 1
        kw = dict(periodic=(1, 0, 1)) if i != 2 else dict(periodic=(0, 1, 0), reservoir_z=1, rho_in=1.001, rho_out=0.999)
        d = lbm.Domain(lab, (0.4 * lab).astype(np.float32), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95,
                       force=(0.0, 0.0, 1e-5), precision=precision, **kw)
        d.init_fluids(np.random.default_rng(i).uniform(-0.9, 0.9, lab.shape))
        doms.append(d)
    return doms


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("grow", [8, 9])         # layers more
def test_by_job_is_the_same(grow, precision):
    import paper_2007_12266_gb300 as lbm
    runs = []
    for shape in (None, (256, -1, -1)):
        doms = _domains(precision, grow)
        b = lbm.Batch()
        for d in doms:
            b.add(d)
        if shape:
            b.set_launch(*shape)
        n0 = b.launch_count
        for steps in (2, 24, 6):                 # no middle steps, bundles of 16 and 2, bundles of 2
            b.advance(steps)
        launches = b.launch_count - n0
        mean = b.n_sites / len(doms)
        # two kernels per step and job, one more for the reservoirs; or per step
        assert launches == 32 * (2 * len(doms) + 1 if not shape and mean >= 80 << 10 else 3)
        m = b.measure()
        runs.append([[d.distributions(k) for k in ("f", "a", "b")] for d in doms] + [m])
        b.close()
        for d in doms:
            d.close()
    for x, y in zip(runs[0][:-1], runs[1][:-1]):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
    assert runs[0][-1] == runs[1][-1]
