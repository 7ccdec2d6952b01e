"""The FP32 build's seeding (short double-precision forms, redone by the
library's functions near a rounding boundary) gives the records of the FP64
build's seeding rounded to float, bit for bit."""
import numpy as np
import pytest

import pic_inputs as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1704_01202_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("T_e,T_i,beam", [(10.0, 10.0, 0.05), (2e4, 300.0, 0.0), (0.0, 0.0, 1.0), (1e-3, 1e-3, 0.5)])
def test_seeded_momenta_are_the_rounded_doubles(tables, T_e, T_i, beam):
    cfg = P.cfg_small_1d(nx=4096, ppc_e=200, ppc_i=40, T_e_eV=T_e, T_i_eV=T_i, beam_frac=beam, seed=77,
                         m_ion_me=float(np.float32(P.M_AL_ME)))     # the same mass in both builds
    got = []
    for fp64 in (False, True):
        s = pkg.Slab(cfg, tables, fp64=fp64)
        s.seed()
        got.append((s.electrons(full=True), s.ions(full=True)))
        s.close()
    for a, b in zip(*got):
        ka, kb = np.argsort(a["id"]), np.argsort(b["id"])
        assert np.array_equal(a["id"][ka], b["id"][kb])
        u = b["u"][kb].astype(np.float32)
        assert np.array_equal(a["u"][ka].astype(np.float32), u)
        assert beam == 1.0 or T_e == 0.0 or np.unique(u).size > u.size // 4
