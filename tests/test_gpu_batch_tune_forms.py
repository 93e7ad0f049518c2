"""A tuned launch shape is kept for batches of the same kind only: where the default
shape means job by job, it is not taken from a batch for which it means one launch per
pass over all jobs, nor the other way round, though both have as many sites (GPU only;
in a process of its own, since the shapes are kept per process)."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import numpy as np
import paper_2007_12266_gb300 as lbm

def batch(edges):
    doms = []
    b = lbm.Batch()
    for e in edges:
        lab = np.zeros((e, e, e), np.uint16)
        d = lbm.Domain(lab, None, tau_a=0.7, tau_b=0.7, alpha=0.005, beta=0.95, force=(0.0, 0.0, 1e-5))
        d.init_fluids(np.full(lab.shape, 0.5, np.float32))
        doms.append(d)
        b.add(d)
    return b, doms

def tuned(edges):
    b, doms = batch(edges)
    n0 = b.launch_count
    shape = b.tune(4)
    n = b.launch_count - n0        # 0: the shape of an earlier batch
    b.close()
    return n, shape

few, many = [50], [20] * 15        # 125,000 and 120,000 sites
for edges in ORDER:
    print(*[tuned(edges) for _ in range(2)], sep="|")
"""


@pytest.mark.parametrize("order", ["[many, few]", "[few, many]"])
def test_shapes_are_kept_by_form(order):
    r = subprocess.run([sys.executable, "-c", PROGRAM.replace("ORDER", order)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [[eval(x) for x in line.split("|")] for line in r.stdout.strip().splitlines()]
    assert len(lines) == 2
    for (n1, shape1), (n2, shape2) in lines:
        assert n1 > 0                          # timed for itself
        assert n2 == 0 and shape2 == shape1    # and kept for the next of its kind
