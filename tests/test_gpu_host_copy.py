"""Large read-backs, whose pages are populated by threads while the copy runs:
whole against the same data read in parts and against plain small copies, into
fresh and into reused memory, at sizes around the threshold and off page and
chunk boundaries (GPU only). The values are copies of device values, so they
are equal bit for bit."""
import ctypes as ct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _domain(nx, ny, nz):
    import paper_2007_12266_gb300 as lbm
    rng = np.random.default_rng(nx)
    lab = (rng.uniform(size=(nz, ny, nx)) < 0.2).astype(np.uint16)
    dom = lbm.Domain(lab, force=(0.0, 0.0, 1e-5))
    dom.init_fluids(rng.uniform(-1, 1, size=lab.shape).astype(np.float32))
    dom.advance(3)
    return dom, lab


# voxels of the dense field: below, at and above 8 MiB (2^21 floats), and several chunks with a ragged tail
@pytest.mark.parametrize("shape", [(127, 128, 128), (128, 128, 128), (131, 129, 127), (163, 179, 191)],
                         ids=lambda s: "x".join(map(str, s)))
def test_fields_and_distributions_come_whole(shape):
    dom, lab = _domain(*shape)
    rho = dom.read_field("rho")
    f = dom.distributions("f")
    assert np.array_equal(np.isnan(rho), lab != 0)
    assert np.abs(f.astype(np.float64).sum(0) - rho[lab == 0]).max() < 1e-6
    nz, ny, nx = lab.shape
    for z in (0, nz // 2, nz - 1):            # the same populations, read plane by plane
        box = dom.read_box("f", (0, 0, z), (nx, ny, z + 1))[:, 0]
        first = int(np.count_nonzero(lab[:z] == 0))
        pore = lab[z] == 0
        assert np.array_equal(box[:, pore], f[:, first:first + int(np.count_nonzero(pore))])
    # into memory that exists already, at an odd offset inside a larger buffer that keeps its other contents
    L, h = dom._L, dom._h
    buf = np.full(f.size + 1000, -7.0, np.float32)
    for off in (0, 333):
        assert L.lbpm_read_distributions(h, 0, ct.c_void_p(buf.ctypes.data + 4 * off)) == 0
        assert np.array_equal(buf[off:off + f.size], f.ravel())
        assert (buf[off + f.size:] == -7.0).all() or off == 333
        buf[:] = -7.0
    dom.close()
