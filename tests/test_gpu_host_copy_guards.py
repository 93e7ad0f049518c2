"""Large read-backs into memory that does not exist yet, beside memory that does: the
pages that threads populate are rounded out to whole ones, and what lies in those before
and behind the result keeps its contents (GPU only)."""
import ctypes as ct
import mmap

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lead", [0, 4, 333 * 4, mmap.PAGESIZE - 4, mmap.PAGESIZE + 1236])   # bytes before the result
def test_neighbours_of_a_fresh_result_keep_their_contents(lead):
    import paper_2007_12266_gb300 as lbm
    rng = np.random.default_rng(5)
    lab = (rng.uniform(size=(96, 101, 97)) < 0.2).astype(np.uint16)
    dom = lbm.Domain(lab, force=(0.0, 0.0, 1e-5))
    dom.init_fluids(rng.uniform(-1, 1, size=lab.shape).astype(np.float32))
    dom.advance(3)
    f = dom.distributions("f")
    assert f.nbytes > 6 << 23                          # several chunks of 8 MiB
    size = 2 * mmap.PAGESIZE + lead + f.nbytes + 2 * mmap.PAGESIZE
    with mmap.mmap(-1, size) as m:                     # anonymous: no page exists
        buf = np.frombuffer(m, np.uint8)
        at = 2 * mmap.PAGESIZE + lead
        before, behind = buf[:at], buf[at + f.nbytes:]
        mark = rng.integers(0, 256, 4096, np.uint8)
        k = min(len(mark), len(before), len(behind))
        before[len(before) - k:] = mark[:k]
        behind[:k] = mark[:k]
        assert dom._L.lbpm_read_distributions(dom._h, 0, ct.c_void_p(buf.ctypes.data + at)) == 0
        assert np.array_equal(buf[at:at + f.nbytes].view(np.float32) if at % 4 == 0 else buf[at:at + f.nbytes],
                              f.ravel() if at % 4 == 0 else f.ravel().view(np.uint8))
        assert np.array_equal(before[len(before) - k:], mark[:k]) and np.array_equal(behind[:k], mark[:k])
        assert not before[:len(before) - k].any() and not behind[k:].any()
        del buf, before, behind
    dom.close()
