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


@pytest.mark.parametrize("ppc_e,ppc_i,T_e", [(31, 1, 10.0), (33, 32, 2e4), (100, 25, 3e5), (128, 128, 30.0),
                                             (129, 31, 30.0), (300, 500, 30.0), (505, 102, 30.0), (600, 130, 50.0)])
def test_team_and_warp_agree(tables, ppc_e, ppc_i, T_e):
    """A slab alone has fewer cells than fill the GPU (a block per cell in the
    cell kernel, staged at the largest size, and in the push); in a context of
    4096 cells the same slab goes one warp per cell through the tiers of its
    sizes.  Same state bit for bit, with created electrons, particles leaving
    through the boundaries and moves of more than a cell (T_e = 3e5)."""
    cfg = P.cfg_small_1d(nx=24, ppc_e=ppc_e, ppc_i=ppc_i, T_e_eV=T_e, flags=P.F_ALL, rad_every=1)
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2, bandwidth_eV=60.0)
    st = _busy(cfg, seed=6)
    ce, ci = pkg.default_capacity(st.n_e, st.n_i, cfg.Z_init)
    one = pkg.Slab(cfg, tables, pl)
    one.load(st)
    many = pkg.Batch(tables, 2, 2048, 2 * ce, 2 * ci)
    slot = many.admit(cfg, st, pl)
    one.step(5)
    many.step(5)
    for a, b in ((one.electrons(), many.electrons(slot)), (one.ions(), many.ions(slot))):
        ka, kb = np.argsort(a["id"]), np.argsort(b["id"])
        for q in a:
            assert np.array_equal(a[q][ka], b[q][kb]), q
    da, db = one.diagnostics(), many.diagnostics(slot)
    assert da["counts"] == db["counts"]
    assert ppc_e != 100 or da["counts"]["ESC_E"] > 0
    one.close()
    many.close()
