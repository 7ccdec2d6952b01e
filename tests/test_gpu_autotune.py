"""The launch-shape search where a cell takes one warp: all four shapes, over
steps that can be compared."""
import numpy as np
import pytest

import pic_inputs as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1704_01202_gb300 as pkg  # noqa: E402


def _slab(rad_every):
    cfg = P.cfg_foil_2d(nx=64, ny=16, rad_every=rad_every)
    pl = P.pulse_foil_2d(I_peak_Wcm2=3e17, fwhm_fs=10.0, t_peak_fs=0.0)
    s = pkg.Slab(cfg, P.standin_tables(), pl)
    s.load(P.init_particles(cfg))
    return s


def _state(s):
    e, i = s.electrons(), s.ions()
    return [d[q][np.argsort(d["id"])] for d in (e, i) for q in sorted(d)]


@pytest.mark.parametrize("rad_every,last", [(5, 9), (2, 15), (1, 8)])
def test_shapes_are_timed_on_steps_of_one_kind(rad_every, last):
    """1 2 4 8 8 4 2 1 warps over the steps without radiation (all of them
    where every step has it), the context's first not timed: with a radiation
    step every five, steps 1-4 and 6-9.  The second time of one warp is
    the last, so the search ends with step `last`, and the state is the same as
    without it."""
    s, ref = _slab(rad_every), _slab(rad_every)
    s.autotune(True)
    s.step(last)                        # steps 0 .. last - 1
    half = s.autotune()[1]
    assert (half > 0).all()             # four shapes, each once at least
    s.step(1)
    w, ms = s.autotune()
    assert ms[0] > half[0] and np.array_equal(ms[1:], half[1:])
    assert ms[[1, 2, 4, 8].index(w)] == ms.min()
    s.step(6)
    assert np.array_equal(s.autotune()[1], ms)
    ref.step(last + 7)
    assert all(np.array_equal(a, b) for a, b in zip(_state(s), _state(ref)))
    s.close()
    ref.close()


def test_steps_of_two_slabs_with_radiation_between():
    """Slabs of one batch at different times: a step is timed when none of
    them has radiation."""
    cfg = P.cfg_small_1d(nx=1024, ppc_e=26, ppc_i=6, flags=P.F_ALL, rad_every=4)
    pl = P.Pulse(I_peak_Wcm2=3e17, fwhm_fs=30.0, t_peak_fs=0.0, hv_eV=1700.0, n_bins=2)
    st = P.init_particles(cfg)
    ce, ci = pkg.default_capacity(st.n_e, st.n_i, cfg.Z_init)
    b = pkg.Batch(P.standin_tables(), 2, 1024, 2 * ce, 2 * ci)
    b.admit(cfg, st, pl)
    b.step(2)
    b.admit(cfg, st, pl)                # two steps behind: radiation every other step
    b.autotune(True)
    seen = []
    for _ in range(16):                 # the second slab's steps 0, 1, ...: 1, 3, 5, ... are timed
        b.step(1)
        seen.append(b.autotune()[1].sum())
    grew = np.diff([0.0] + seen) > 0
    assert grew.tolist() == [k % 2 == 1 for k in range(16)]
    b.close()
