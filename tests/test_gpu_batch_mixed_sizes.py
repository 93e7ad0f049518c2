"""Batches of jobs of very different sizes (GPU only): many small jobs among a large one
are advanced by one launch per pass over all jobs, although the mean size alone would
have the jobs run one by one (for a few small ones they do); the results are the same
bit for bit as with a launch shape that never runs job by job."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _domain(edge, seed, precision):
    import paper_2007_12266_gb300 as lbm
    lab = np.zeros((edge, edge, edge), np.uint16)
    lab[::5, ::6, ::7] = 1
    d = lbm.Domain(lab, (0.4 * lab).astype(np.float32), tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95,
                   force=(0.0, 0.0, 1e-5), precision=precision, periodic=(1, 0, 1))
    d.init_fluids(np.random.default_rng(seed).uniform(-0.9, 0.9, lab.shape))
    return d


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("edges, by_job", [([100] + [20] * 11, False), ([100] + [20] * 2, True), ([20] * 3, False)],
                         ids=["many-small", "few-small", "small"])
def test_mixed_sizes(edges, by_job, precision):
    import paper_2007_12266_gb300 as lbm
    runs = []
    for shape in (None, (256, -1, -1)):
        doms = [_domain(e, i, precision) for i, e in enumerate(edges)]
        b = lbm.Batch()
        for d in doms:
            b.add(d)
        if shape:
            b.set_launch(*shape)
        n0 = b.launch_count
        b.advance(24)
        launches = b.launch_count - n0
        assert launches == 24 * 2 * (len(doms) if by_job and not shape else 1)
        b.measure()
        runs.append([[d.distributions(k) for k in ("f", "a", "b")] for d in doms])
        b.close()
        for d in doms:
            d.close()
    for x, y in zip(*runs):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
