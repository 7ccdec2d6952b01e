"""The 1D field update on both sides of its launch rule: a block per slab up
to a width, grid-wide launches beyond, alone and in batch slots."""
import numpy as np
import pytest

import pic_inputs as P

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


def _cfg(nx, **kw):
    base = dict(nx=nx, dx_nm=2.0, dy_nm=2.0, ppc_e=4, ppc_i=2, T_e_eV=2e3, seed=nx, flags=P.F_PUSH | P.F_FIELD)
    return P.SlabConfig(**{**base, **kw})


def _launches(make, nx):
    """Launches of the field update and the end of a step: a step with
    fields against one without."""
    n = []
    for flags in (P.F_PUSH, P.F_PUSH | P.F_FIELD):
        cfg = _cfg(nx, flags=flags)
        h = make(cfg, P.init_particles(cfg))
        h.use_graphs(False)
        h.step(1)
        n.append(h.launches)
        h.close()
    return n[1] - n[0]


@pytest.mark.parametrize("batch", [False, True])
def test_wide_slabs_are_updated_by_the_whole_grid(tables, batch):
    """A narrow slab's fields and step end take one launch in the place of
    the step end's own.  A wide one is not left to a block: three launches
    over all points, the last with the step end, which a batch has apart."""
    def make(cfg, st):
        if not batch:
            s = pkg.Slab(cfg, tables)
            s.load(st)
            return s
        b = pkg.Batch(tables, 2, cfg.nx, 2 * st.n_e + 64, 2 * st.n_i + 64)
        b.admit(cfg, st)
        return b

    assert _launches(make, 128) == 0
    assert _launches(make, 8192) == (3 if batch else 2)


@pytest.mark.parametrize("nx", [2, 510, 511, 512, 1022, 1023, 1024, 2047, 2048, 4097, 8192])
def test_fields_1d_against_oracle(tables, nx):
    """Two steps in random fields.  Bounds as for one step of every process
    (test_gpu_parity): 1e-5 of the largest field, 2e-5 of the largest
    current; at 2 keV an electron moves a quarter of a cell a step, so the
    FP32 rounding of a position is a few 1e-7 of its current."""
    cfg = _cfg(nx)
    st = P.init_particles(cfg)
    f = P.random_fields(cfg, 3, e_amp=2e-3, b_amp=2e-3)
    g, o = pkg.Slab(cfg, tables), oracle.OracleSlab(cfg, tables)
    for s in (g, o):
        s.load(st)
        s.set_fields(f)
        s.step(2)
    fg, fo = g.fields(), o.fields()
    for k in fg:
        assert np.abs(fg[k] - fo[k]).max() < 1e-5 * (np.abs(fo[k]).max() + 1e-12), k
    jg, jo = g.current(), o.current()
    for c in range(3):
        assert np.abs(jg[c] - jo[c]).max() < 2e-5 * (np.abs(jo[c]).max() + 1e-12), c
    assert g.diagnostics()["t_fs"] == pytest.approx(2 * cfg.dt_fs)
    g.close()


@pytest.mark.parametrize("slot_cells", [1023, 1024, 8192])
def test_fields_in_wide_batch_slots(tables, slot_cells):
    """Slabs narrower than their slots, one of them retired half way: each
    the same bits as alone, its step count too."""
    cfgs = [_cfg(nx, ppc_e=6, ppc_i=2, seed=nx) for nx in (300, slot_cells, 700)]
    sts = [P.init_particles(c) for c in cfgs]
    b = pkg.Batch(tables, 4, slot_cells, 4 * max(s.n_e for s in sts), 4 * max(s.n_i for s in sts))
    slots = [b.admit(c, s) for c, s in zip(cfgs, sts)]
    b.step(3)
    b.retire(slots[2])
    b.step(4)
    for cfg, st, k in zip(cfgs[:2], sts, slots):
        one = pkg.Slab(cfg, tables)
        one.load(st)
        one.step(7)
        for a, c in ((one.electrons(), b.electrons(k)), (one.ions(), b.ions(k))):
            ka, kc = np.argsort(a["id"]), np.argsort(c["id"])
            for q in a:
                assert np.array_equal(a[q][ka], c[q][kc]), q
        assert b.slot(k)[1] == 7
        one.close()
    b.close()
