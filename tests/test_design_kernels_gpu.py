"""The design-E kernels and the one-launch E phase, FP32, on either side of the lines between them, against the
FP64 oracle: pairable and odd boxes, grids whose E phase is one round of blocks or more, columns of one and two
planes, with each of the pole loops.  Tolerances: the method's."""
import pytest

import synth
from synth import base_desc, vacuum
from test_parity_gpu import compare, gpu, run_oracle  # noqa: F401
from test_step_layout_gpu import run

pytestmark = pytest.mark.gpu


# E phase of one round: 48^3, 64 x 64 x 32, 34^3 (one-cell shell kernels); of two: 64 x 48 x 48; odd x start of the box.
# Columns of two planes, an odd number of planes: 64^3 (two planes make it one round).
@pytest.mark.parametrize("poles", [0, 3, 7])
@pytest.mark.parametrize("n,design", [((48, 48, 48), (24, 24, 24)), ((64, 64, 32), (30, 30, 12)), ((34, 34, 34), (12, 10, 8)),
                                      ((64, 48, 48), (44, 28, 30)), ((47, 44, 40), (21, 20, 18)),
                                      ((48, 46, 52), (32, 32, 38)), ((50, 46, 52), (34, 32, 38)),
                                      ((64, 64, 64), (32, 32, 31))])
def test_design_kernels(gpu, n, design, poles):  # noqa: F811
    d = base_desc(*n, n_steps=70, cpml=5, design=design, gap=(2, 2, 2), src_kind=0, src_comp=1, src_pos=(n[0] // 2, 6, n[2] - 7))
    d["src_t0"], d["src_fwhm_hz"], d["adj_tau"] = 20 * d["courant"] * d["dx"] / synth.C0, 2e15, 1.5e-16
    m2 = synth.drude_lorentz_metal(poles, poles) if poles else synth.lorentz_dielectric(3, 0)
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=m2, gamma=0.0, rho=synth.smooth_rho(synth.box_shape(d["design_box"]), 5, 2.0))
    compare(run(gpu, w, 1), run_oracle(w), 32)
