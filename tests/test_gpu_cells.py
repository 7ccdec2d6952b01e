"""The cell kernel at the sizes where its path changes: cells of one warp
(sorted in registers up to 32, 64, 128, 256 and 512 entries) and of a block
of four warps (shares of 32 to 512 entries a warp, merged by rank), against
numpy's order and, one step of every process, against the FP64 oracle with
the parity bounds of test_gpu_parity."""
import numpy as np
import pytest

import pic_inputs as P
from test_gpu_parity import _assert_parity, _busy, _run_both

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_1704_01202_gb300 as pkg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    pkg.build()
    oracle.build()


@pytest.mark.parametrize("n", [1, 32, 33, 65, 127, 128, 255, 256, 257, 511, 512, 513, 1023, 1025, 2047, 2048, 2049, 4096])
@pytest.mark.parametrize("top_bits", [0, 3, 18, 64])
def test_cell_order_at_share_edges(n, top_bits):
    """Ascending (key, id) whatever the keys share: nothing (64), all but
    their low bits, or (18 and 3 random top bits, the rest from a few values)
    the bits the sort's words carry, so that whole runs are decided by the
    low words and the ids."""
    rng = np.random.default_rng(100 * n + top_bits)
    ids = rng.permutation(np.arange(7 * n, dtype=np.uint64))[:n] * np.uint64(0x100000001)
    if top_bits == 64:
        key = rng.integers(0, 2**64 - 1, n, dtype=np.uint64, endpoint=True)
    else:
        key = rng.integers(0, 3, n, dtype=np.uint64)
        if top_bits:
            key |= rng.integers(0, 1 << top_bits, n, dtype=np.uint64) << np.uint64(64 - top_bits)
    ref = np.lexsort((ids, key))
    for rmax in (128, 512, 1024):
        if rmax == 128 and n > 128:
            continue
        assert np.array_equal(pkg.order_check(key, ids, rmax), ref), rmax


@pytest.mark.parametrize("ppc_e,ppc_i", [(32, 33), (128, 128), (129, 31), (40, 130), (255, 16), (512, 102), (513, 128),
                                         (300, 512), (1025, 256), (2000, 500)])
def test_cell_sizes_one_step(tables, ppc_e, ppc_i):
    cfg = P.cfg_small_1d(nx=5, ppc_e=ppc_e, ppc_i=ppc_i, T_e_eV=40.0, flags=P.F_ALL, rad_every=1)
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2, bandwidth_eV=60.0)
    st = _busy(cfg, seed=4)
    g, o = _run_both(cfg, tables, st, 1, pulse=pl, photons=P.photons_uniform(cfg, pl, 0.5))
    _assert_parity(cfg, st, g, o)
