"""The blocked DFT kernel where its blocks end: design boxes whose 3 nd samples fill its 512-sample chunks
exactly, leave a ragged or tiny last chunk, or give snapshot slots that need padding to 16 bytes (every
nd mod 4), with full and partial 16-step blocks and one to eight frequencies, element by element against the
FP64 oracle.  Tolerances: the method's, 1e-4 (FP32 fields) and 1e-10 (FP64)."""
import numpy as np
import pytest

import synth
from parity_util import TOL, rel
from synth import base_desc, vacuum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("design,nf,steps", [((8, 8, 8), 3, 32), ((8, 8, 8), 8, 37), ((5, 5, 5), 1, 7), ((6, 7, 9), 2, 50),
                                             ((9, 9, 15), 3, 17), ((7, 10, 5), 3, 48)])
def test_dft_block_ends(design, nf, steps, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2305_00234_gb300 import build
    build.build()
    import paper_2305_00234_gb300 as lib
    d = base_desc(24, 22, 26, n_steps=steps, cpml=4, precision=prec, design=design, gap=(2, 2, 2),
                  lambdas_nm=tuple(np.linspace(400.0, 900.0, nf)), src_pos=(12, 11, 13))
    d["src_t0"] = 0.3 * steps * d["courant"] * d["dx"] / synth.C0
    d["src_fwhm_hz"] = 1.2e16 / steps * 10
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(5, 2), gamma=0.0,
             rho=synth.uniform_rho(synth.box_shape(d["design_box"]), 9))
    p, o = lib.problem(w), oracle.problem(w)
    Fg, _ = p.forward()
    Fo, _ = o.forward()
    a, b = p.dft(), o.get_dft()
    p.close()
    o.close()
    assert abs(Fg - Fo) <= TOL[prec] * abs(Fo)
    for f in range(nf):
        for c in range(3):
            assert rel(a[f, c], b[f, c]) <= TOL[prec], (f, c, rel(a[f, c], b[f, c]))
