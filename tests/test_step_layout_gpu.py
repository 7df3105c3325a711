"""The background step by the shell kernels on the whole grid and by the interior kernel with the shell around it,
whichever of the two the grid's size would select (fdtd_set_step_layout): both against the FP64 oracle, and
against each other, at the edges the split and the launch shapes have: interior boxes whose x start falls on
each alignment, partial tiles, columns of every depth, blocks of both sizes.  Tolerances: the method's."""
import pytest

import synth
from parity_util import TOL, rel
from synth import base_desc, vacuum
from test_parity_gpu import compare, gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def run(lib, w, layout):
    p = lib.problem(w)
    p.set_step_layout(layout)
    F, gap = p.forward()
    g = {"F": F, "gap": gap, "fields": [p.field(c) for c in range(6)], "dft": p.dft(),
         "maps": [p.index_map(q) for q in range(4)], "p": p}
    p.adjoint()
    g["adft"], g["grad"] = p.dft(True), p.gradient()
    return g


# the inputs of test_step_paths, which the interior kernel's box splits raggedly in all three tile axes: x rows of 52
# and 72 cells (no multiple of 128 bytes: x start on 32 bytes), 96 (on 128 bytes), 64 (too narrow for that: 32 bytes)
@pytest.mark.parametrize("src", ["tfsf", "dipole_shell", "dipole_interior"])
@pytest.mark.parametrize("prec,nx", [(32, 52), (32, 64), (32, 72), (32, 96), (64, 46), (64, 72)])
def test_both_layouts_against_the_oracle(gpu, prec, nx, src):  # noqa: F811
    kw = {"tfsf": dict(src_kind=1, src_pos=(9, 0, 0)), "dipole_shell": dict(src_kind=0, src_comp=1, src_pos=(8, 33, 6)),
          "dipole_interior": dict(src_kind=0, src_comp=2, src_pos=(12, 8, 8))}[src]
    d = base_desc(nx, 42, 37, n_steps=420, cpml=(6, 5, 4, 7, 5, 3), precision=prec, design=(22, 18, 15), gap=(2, 2, 2),
                  lambdas_nm=(500.0, 650.0), **kw)
    rho = synth.smooth_rho(synth.box_shape(d["design_box"]), 23, 2.0)
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(23, 3), gamma=1e6, rho=rho)
    o = run_oracle(w)
    a, b = run(gpu, w, 1), run(gpu, w, 2)
    assert a["p"].timings()["interior_cells"] == 0 and b["p"].timings()["interior_cells"] > 0
    for g in (a, b):
        compare(g, o, prec)
    for x, y in zip(a["fields"], b["fields"]):
        assert rel(x, y) <= TOL[prec]


# launches of few blocks (short columns, blocks of 128), of about one round and of several; odd rows (one-cell kernels)
@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [(12, 10, 9), (24, 96, 10), (46, 34, 75), (45, 33, 70), (64, 96, 40)])
def test_shell_shapes(gpu, n, prec):  # noqa: F811
    d = base_desc(*n, n_steps=60, cpml=2, precision=prec, design=(4, 4, 4), gap=(2, 2, 2), src_kind=0, src_comp=1,
                  src_pos=(n[0] // 2, 3, n[2] - 3))
    d["src_t0"], d["src_fwhm_hz"], d["adj_tau"] = 20 * d["courant"] * d["dx"] / synth.C0, 2e15, 1.5e-16
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(3, 1), gamma=0.0,
             rho=synth.uniform_rho(synth.box_shape(d["design_box"]), 3))
    compare(run(gpu, w, 1), run_oracle(w), prec)


def test_layout_errors(gpu):  # noqa: F811
    d = base_desc(12, 12, 12, n_steps=20, cpml=2, design=(4, 4, 4), gap=(2, 2, 2))
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(3, 1), gamma=0.0,
             rho=synth.uniform_rho((4, 4, 4), 3))
    p = gpu.problem(w)
    for bad in (-1, 3, 2):                             # 2: no interior box on this grid
        with pytest.raises(gpu.FdtdError):
            p.set_step_layout(bad)
    p.set_step_layout(1)
    p.forward()
    p.close()
