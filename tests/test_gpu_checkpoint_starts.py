"""A checkpoint image whose cell starts are damaged is refused and the slab keeps
its state."""
import numpy as np
import pytest

import pic_inputs as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1704_01202_gb300 as pkg  # noqa: E402

HEADER = 8 + 6 * 4 + 2 * 8 + 2 * 4 + 4 * 8 + 2 * 8


def test_damaged_cell_starts(tables):
    cfg = P.cfg_small_1d(nx=16, ppc_e=16, ppc_i=4)
    s = pkg.Slab(cfg, tables)
    s.load(P.init_particles(cfg))
    s.step(2)
    image = s.checkpoint()
    ne, ni = s.counts()
    at = HEADER + 32 * (ne + ni)
    starts = np.frombuffer(image, dtype=np.int32, count=2 * (cfg.nx + 1), offset=at)
    assert starts[0] == 0 and starts[cfg.nx] == ne and starts[cfg.nx + 1] == 0 and starts[-1] == ni
    for k in (3, cfg.nx + 1 + 3):
        for value in (starts[k + 1] + 1, ne + ni + 100000, -1):
            bad = np.array(starts)
            bad[k] = value
            with pytest.raises(pkg.PicError, match="ARG"):
                s.restore(image[:at] + bad.tobytes() + image[at + bad.nbytes:])
    s.restore(image)
    assert s.counts() == (ne, ni)
    s.close()
