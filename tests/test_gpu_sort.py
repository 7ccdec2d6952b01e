"""The counting sort where its launches change: cell counts around a scan
tile (4096) and around the most tiles one launch scans by itself (8), with
empty cells, groups that span cells, and particles that leave."""
import numpy as np
import pytest

import pic_inputs as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1704_01202_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(2, 1), (31, 1), (4095, 1), (4096, 1), (4097, 1), (4096, 8), (4099, 8), (8192, 5)])
def test_sorted_after_free_streaming(tables, nx, ny):
    """Push alone, without fields: straight lines, known to FP32 rounding; the
    library's order is cell by cell with every particle in its own cell, and
    every id that did not leave is there once."""
    rng = np.random.default_rng(nx + ny)
    cfg = P.SlabConfig(nx=nx, ny=ny, dx_nm=2.0, dy_nm=2.0, ppc_e=3, ppc_i=1, T_e_eV=2e4, T_i_eV=1e6, seed=5, flags=P.F_PUSH)
    st = P.init_particles(cfg)
    keep = rng.random(st.n_e) < 0.6                      # uneven and empty cells
    st = P.ParticleState(eX=st.eX[keep], eY=st.eY[keep], eu=st.eu[keep], ew=st.ew[keep], eid=st.eid[keep], iX=st.iX,
                         iY=st.iY, iu=st.iu, izf=st.izf, iZ=st.iZ, inK=st.inK, iid=st.iid)
    s = pkg.Slab(cfg, tables)
    s.load(st)
    steps = 3
    s.step(steps)
    for got, X, Y, u, ids in ((s.electrons(), st.eX, st.eY, st.eu, st.eid), (s.ions(), st.iX, st.iY, st.iu, st.iid)):
        v = u / np.sqrt(1.0 + (u ** 2).sum(1))[:, None] * (299.792458 * cfg.dt_fs / cfg.dx_nm) * steps
        x = X + v[:, 0]
        y = (Y + v[:, 1]) % ny if ny > 1 else Y
        # at the boundaries, rounding decides who has left
        inside, outside = (x > 1e-4) & (x < nx - 1e-4), (x < -1e-4) | (x > nx + 1e-4)
        assert np.unique(got["id"]).size == got["id"].size
        assert np.isin(ids[inside], got["id"]).all() and not np.isin(ids[outside], got["id"]).any()
        k = np.searchsorted(ids, got["id"])
        assert np.array_equal(ids[k], got["id"])
        assert np.abs(got["X"] - x[k]).max(initial=0.0) < 1e-4
        dy = np.abs(got["Y"] - y[k])
        assert np.minimum(dy, ny - dy).max(initial=0.0) < 1e-4 if ny > 1 else not dy.any()
        cell = np.floor(got["Y"]).astype(int) * nx + np.floor(got["X"]).astype(int) if ny > 1 else np.floor(got["X"]).astype(int)
        assert (np.diff(cell) >= 0).all()
    s.close()
