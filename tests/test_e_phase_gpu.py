"""Which form the E phase of a step takes, and its results against the FP64 oracle, beside paired shell kernels (FP32, even
x CPML): one launch or two, seen in the launch count; the paired and the one-sample design kernel; columns of one and of
two planes; each of the pole loops.  Tolerances: the method's."""
import pytest

import synth
from synth import base_desc, vacuum
from test_parity_gpu import compare, gpu, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu

STEPS = 420   # of test_paired_design_paths, as the pulse and the wavelengths are


# one launch: up to four poles, shell columns of one plane, and with the one-sample design kernel at most one round of
# blocks (60^3 has 1.35); 64^3: design columns of two planes make it one round; 72^3: shell columns of two planes
@pytest.mark.parametrize("poles", [0, 3, 7])
@pytest.mark.parametrize("n,design,paired,one", [((48, 48, 48), (24, 24, 24), 1, True), ((48, 48, 48), (21, 24, 24), 0, True),
                                                 ((64, 64, 64), (32, 32, 31), 1, True), ((44, 50, 54), (22, 24, 28), 0, True),
                                                 ((60, 60, 60), (31, 31, 31), 0, False), ((72, 72, 72), (36, 36, 36), 1, False)])
def test_e_phase_form(gpu, n, design, paired, one, poles):  # noqa: F811
    d = base_desc(*n, n_steps=STEPS, cpml=6, design=design, gap=(2, 2, 2), lambdas_nm=(500.0, 650.0), src_kind=0, src_comp=1,
                  src_pos=(n[0] // 2, 7, n[2] - 8))
    m2 = synth.drude_lorentz_metal(poles, poles) if poles else dict(vacuum(), eps_inf=[2.0, 2.25, 2.5])
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=m2, gamma=0.0, rho=synth.smooth_rho(synth.box_shape(d["design_box"]), 5, 2.0))
    g = run_gpu(gpu, w)
    t = g["p"].timings()
    assert t["paired_shell"] == 1 and t["paired_design"] == paired and t["interior_cells"] == 0
    before = t["launches"]
    F, _ = g["p"].forward()
    assert F == g["F"]
    per_step = 2 if one and poles <= 4 else 3           # H, E or shell E and design E
    blocks = (STEPS + 15) // 16                        # each with its DFT and the two launches that begin and end it
    assert g["p"].timings()["launches"] - before == per_step * STEPS + 3 * blocks + 1
    compare(g, run_oracle(w), 32)
    g["p"].close()
