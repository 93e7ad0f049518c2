"""The neighbour records of the step kernels (ranks of the eight rows next to a
site) against the FP64 oracle, at the shapes where a record can fail: rows of
one and two voxels, sites next to a periodic x face (whose neighbours are
looked up in the dense grid of ids), warps that mix both, ragged last warps, and
rows so long that a rank difference exceeds 16 bits (GPU only).

Tolerance: each fp32 timestep keeps every distribution within 1e-6
max(|o|, w_q) of the oracle's; a call of k steps is held to k times that.
"""
import numpy as np
import pytest

from lbm_cases import compare_state, pair, random_state, set_both
from synthetic import random_affinity, sphere_pack

pytestmark = pytest.mark.gpu

KW = dict(tau_a=0.8, tau_b=0.65, alpha=0.01, beta=0.8, force=(1e-5, -2e-5, 3e-5))

SHAPES = [(1, 5, 7), (2, 4, 6), (31, 6, 5), (32, 5, 6), (33, 4, 7), (70, 6, 6)]


def _image(nx, ny, nz):
    if min(nx, ny, nz) < 4:
        lab = (np.random.default_rng(nx).uniform(size=(nz, ny, nx)) < 0.3).astype(np.uint16)
        lab[0, 0, 0] = 0
        return lab
    return sphere_pack((nx, ny, nz), 0.5, 1.6, 0.4, 7 + nx).labels


@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 1), (1, 0, 0), (0, 0, 0)], ids=["ppp", "wpp", "pww", "www"])
@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_steps_match_oracle(shape, periodic):
    lab = _image(*shape)
    aff = random_affinity(lab, -0.9, 0.9, 11)
    for start in (0, 1):
        dom, ref = pair(lab, aff, periodic, **KW)
        sv, nb = dom.index()
        sv_o, nb_o = ref.index()
        assert np.array_equal(sv, sv_o) and np.array_equal(nb, nb_o)
        set_both(dom, ref, random_state(ref, seed=5 + start), start)
        for k in (1, 3):                    # population form, then a call in the sum form
            dom.advance(k)
            ref.step(k)
        assert max(compare_state(dom, ref)) <= 4e-6
        dom.close()


def test_rank_differences_beyond_16_bits():
    """Rows of 36,000 open voxels: the rank of the next row is that far away."""
    lab = np.zeros((3, 4, 36000), np.uint16)
    lab[:, 0, ::7] = 1
    lab[1, 2, 5::11] = 1
    aff = random_affinity(lab, -0.5, 0.5, 3)
    dom, ref = pair(lab, aff, (0, 1, 1), **KW)
    set_both(dom, ref, random_state(ref, seed=9), 0)
    dom.advance(3)
    ref.step(3)
    assert max(compare_state(dom, ref)) <= 3e-6
    dom.close()
