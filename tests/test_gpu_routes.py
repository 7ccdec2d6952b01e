"""Routes of the cell kernel that a small slab alone does not take: the chain
of tiers and the look-ahead instance belong to contexts of many cells (a
team of warps takes each cell of the others); and the cell sums with a bulk
limit, by a team and by one warp."""
import numpy as np
import pytest

import pic_inputs as P
from parity_util import match, momentum_errors
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


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _one_warp_cells():
    """More cells than a context whose cells take a team of four warps has."""
    return 4 * _sms() + 90


def _uneven(cfg, extra):
    """The configuration's particles, and in the cells of `extra` (electrons,
    ions) more."""
    st = P.init_particles(cfg)
    rng = np.random.default_rng(9)
    eX, eu, ew, iX, iu = [st.eX], [st.eu], [st.ew], [st.iX], [st.iu]
    for c, (ne, ni) in extra.items():
        eX.append(c + P._f32(rng.random(ne) * 0.999))
        eu.append(P._f32(rng.standard_normal((ne, 3)) * 0.01))
        ew.append(np.full(ne, st.ew[0]))
        iX.append(c + P._f32(rng.random(ni) * 0.999))
        iu.append(P._f32(rng.standard_normal((ni, 3)) * 1e-5))
    n_e, n_i = (sum(x.size for x in v) for v in (eX, iX))
    return P.ParticleState(
        eX=np.concatenate(eX), eY=np.full(n_e, 0.5), eu=np.concatenate(eu), ew=np.concatenate(ew),
        eid=np.arange(n_e, dtype=np.uint64), iX=np.concatenate(iX), iY=np.full(n_i, 0.5), iu=np.concatenate(iu),
        izf=np.zeros(n_i), iZ=np.full(n_i, cfg.Z_init, dtype=np.int32), inK=np.zeros(n_i, dtype=np.int32),
        iid=np.arange(n_i, dtype=np.uint32))


def _same_state(one, many, k):
    for a, b in ((one.electrons(), many.electrons(k)), (one.ions(), many.ions(k))):
        ka, kb = np.argsort(a["id"]), np.argsort(b["id"])
        for q in a:
            assert np.array_equal(a[q][ka], b[q][kb]), q
    counts = one.diagnostics()["counts"]
    assert counts == many.diagnostics(k)["counts"]
    return counts


@pytest.mark.parametrize("extra,tiers", [({}, 0), ({5: (60, 20), 17: (10, 40)}, 1), ({5: (300, 90), 640: (500, 40)}, 1),
                                         ({5: (300, 90), 17: (500, 40), 40: (1500, 400)}, 2)])
def test_uneven_cells_chain_of_tiers(tables, extra, tiers):
    """Most cells staged by the first tier, a few too large for it and one for
    the next: one warp a cell, then a team.  The launches of a step tell which
    tiers ran: one more each than for even cells."""
    cfg = P.cfg_small_1d(nx=_one_warp_cells(), ppc_e=24, ppc_i=6, T_e_eV=30.0, flags=P.F_ALL & ~P.F_PHOTO)
    launches = []
    for ex in ({}, extra):
        st = _uneven(cfg, ex)
        s = pkg.Slab(cfg, tables, cap_e=st.n_e + 13 * st.n_i, cap_i=st.n_i + 64)
        s.use_graphs(False)
        s.load(st)
        s.step(1)
        launches.append(s.launches)
        s.close()
    assert launches[1] - launches[0] == tiers
    g, o = _run_both(cfg, tables, st, 1)
    _assert_parity(cfg, st, g, o)


BULK = [(5, 100, 25), (5, 700, 102), (0, 33, 8), (0, 100, 25)]


@pytest.mark.parametrize("nx,ppc_e,ppc_i", BULK)
def test_bulk_limit_fp64(tables, nx, ppc_e, ppc_i):
    """E_bulk > 0: temperature, recombination and its energy payment over the
    electrons below it alone.  A rad step of every process in the FP64 build,
    whose arithmetic is the oracle's but for rounding; nx 0: a context whose
    cells take a warp each.  A sum over other electrons would move every
    momentum of a cell by parts in a thousand; rounding moves a few by more
    than 1e-12 (near-equal velocities, a slow electron hit by a fast one), none
    by 1e-9.  Weights: the cell's sum (about 4) in 700 additions, 3e-13."""
    cfg = P.cfg_small_1d(nx=nx or _one_warp_cells(), ppc_e=ppc_e, ppc_i=ppc_i, T_e_eV=40.0, E_bulk_eV=75.0, flags=P.F_ALL,
                         rad_every=1)
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2, bandwidth_eV=60.0)
    st = _busy(cfg, seed=4)
    g, o = pkg.Slab(cfg, tables, pl, fp64=True), oracle.OracleSlab(cfg, tables, pl)
    for s in (g, o):
        s.load(st)
        s.set_photons(P.photons_uniform(cfg, pl, 0.5))
        s.step(1)
    ge, oe, gi, oi = g.electrons(full=True), o.electrons(), g.ions(full=True), o.ions()
    ia, ib, same = match(ge["id"], oe["id"])
    ja, jb, same_i = match(gi["id"], oi["id"])
    assert same and same_i
    du = momentum_errors(ge["u"][ia], oe["u"][ib])
    assert np.quantile(du, 0.999) < 1e-12 and du.max() < 1e-9, (np.quantile(du, 0.999), du.max())
    assert np.abs(ge["w"][ia] - oe["w"][ib]).max() < 1e-12
    assert np.array_equal(gi["Z"][ja], oi["Z"][jb]) and np.array_equal(gi["nK"][ja], oi["nK"][jb])
    _, co = o.tallies()
    assert g.diagnostics()["counts"] == co
    assert co["REC"] > 0 and co["ION"] > 0
    g.close()


@pytest.mark.parametrize("ppc_e,ppc_i", [(33, 8), (100, 25), (300, 60), (600, 130)])
def test_bulk_limit_team_and_warp_agree(tables, ppc_e, ppc_i):
    """The same bits from a team a cell (a slab alone) and from the tiers of a
    context of 4096 cells."""
    cfg = P.cfg_small_1d(nx=24, ppc_e=ppc_e, ppc_i=ppc_i, T_e_eV=40.0, E_bulk_eV=75.0, flags=P.F_ALL, rad_every=2)
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2, bandwidth_eV=60.0)
    st = _busy(cfg, seed=6)
    ce, ci = pkg.default_capacity(st.n_e, st.n_i, cfg.Z_init)
    one = pkg.Slab(cfg, tables, pl)
    one.load(st)
    many = pkg.Batch(tables, 2, 2048, 2 * ce, 2 * ci)
    k = many.admit(cfg, st, pl)
    one.step(4)
    many.step(4)
    _same_state(one, many, k)
    one.close()
    many.close()


@pytest.mark.parametrize("slot_cells", [2045, 2048])
def test_look_ahead_agrees(tables, slot_cells):
    """Beyond eight rounds of the resident warps (16 an SM) over the cells,
    cells of at most 128 entries go through the instance that claims its next
    cells early.  Small slabs in the slots of such a batch, and one as wide as
    its slot, against each alone (a team a cell, or the plain instance): the
    same bits over rad steps with created electrons and particles leaving.
    2045: a last round of fewer cells than warps."""
    slots = 8 * 16 * _sms() // slot_cells + 2
    assert slots * slot_cells >= 8 * 16 * _sms()
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2, bandwidth_eV=60.0)
    shapes = [(24, 31, 1, 10.0), (24, 33, 32, 2e4), (24, 90, 23, 3e5), (24, 64, 16, 30.0), (slot_cells, 24, 6, 100.0)]
    cfgs = [P.cfg_small_1d(nx=nx, ppc_e=e, ppc_i=i, T_e_eV=T, flags=P.F_ALL, rad_every=1, seed=k)
            for k, (nx, e, i, T) in enumerate(shapes)]
    sts = [_busy(c, seed=6) for c in cfgs]
    caps = [pkg.default_capacity(s.n_e, s.n_i, c.Z_init) for c, s in zip(cfgs, sts)]
    many = pkg.Batch(tables, slots, slot_cells, sum(e for e, _ in caps), sum(i for _, i in caps))
    at = [many.admit(c, s, pl) for c, s in zip(cfgs, sts)]
    many.step(5)
    ion = 0
    for cfg, st, k in zip(cfgs, sts, at):
        one = pkg.Slab(cfg, tables, pl)
        one.load(st)
        one.step(5)
        ion += _same_state(one, many, k)["ION"]
        one.close()
    assert ion > 0
    many.close()
