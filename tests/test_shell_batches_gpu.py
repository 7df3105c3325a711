"""The FP32 one-cell shell kernels with two z planes a batch of loads, which grids of 2.5 M cells and up take (odd x rows
or an odd x CPML: no cell pairs), against the FP64 oracle on the whole grid: the whole grid by the shell kernels, and the
shell around an interior box.  A pulse beside the low x, y CPML reaches the design box, the slabs and both planes of a
batch in the window; the z extents leave columns that end within a batch.  Tolerances: the method's."""
import pytest

import synth
from synth import base_desc, vacuum
from test_parity_gpu import compare, gpu, run_oracle  # noqa: F401
from test_step_layout_gpu import run

pytestmark = pytest.mark.gpu


# the smallest such grids with an odd and an even z extent; with an interior box (3.9 M of 5.5 M cells; a larger grid)
@pytest.mark.parametrize("n,cpml,interior", [((151, 130, 129), 5, False), ((131, 98, 196), 4, False), ((192, 170, 169), 5, True),
                                              ((232, 200, 197), 5, True)])
def test_two_plane_batches(gpu, n, cpml, interior):  # noqa: F811
    assert n[0] * n[1] * n[2] >= 2500000
    d = base_desc(*n, n_steps=60, cpml=cpml, src_kind=0, src_comp=1, src_pos=(13, 8, 60))
    d["design_box"], d["gap_box"] = [8, 14, 9, 15, 55, 61], [10, 12, 11, 13, 57, 59]
    d["src_t0"], d["src_fwhm_hz"], d["adj_tau"] = 20 * d["courant"] * d["dx"] / synth.C0, 2e15, 1.5e-16
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(3, 1), gamma=0.0,
             rho=synth.uniform_rho(synth.box_shape(d["design_box"]), 3))
    g = run(gpu, w, 0)
    t = g["p"].timings()
    assert t["paired_shell"] == 0 and (t["interior_cells"] > 0) == interior
    compare(g, run_oracle(w), 32)
    g["p"].close()


# one-cell shells take an interior kernel from a box of 3 M cells on, paired ones from grids of 9 M cells on
@pytest.mark.parametrize("n,cpml,box", [((160, 160, 160), 5, 0), ((176, 176, 176), 5, 160 * 160 * 165), ((176, 176, 176), 4, 0)])
def test_layout_line_of_one_cell_shells(gpu, n, cpml, box):  # noqa: F811
    d = base_desc(*n, n_steps=20, cpml=cpml, design=(4, 4, 4), gap=(2, 2, 2))
    p = gpu.Problem(d, vacuum(), vacuum(), synth.drude_lorentz_metal(3, 1))
    assert p.timings()["interior_cells"] == box
    p.close()
