"""Small grids with the interior kernel and its two buffers of every field (fdtd_set_step_layout 2), which by their size the
shell kernels would take whole: the parity cases written for that kernel, paper mode with checkpoints of alternating
buffers, fields after odd numbers of steps, and one handle that changes between the layouts.  Tolerances: the
method's; between checkpoint intervals those of test_paper_graphs_gpu."""
import numpy as np
import pytest

import synth
import test_parity_gpu as parity
from parity_util import TOL, rel
from synth import base_desc, vacuum
from test_paper_mode_gpu import _case, _oracle
from test_parity_gpu import compare, gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def problem(lib, w, layout):
    p = lib.problem(w)
    p.set_step_layout(layout)
    assert (p.timings()["interior_cells"] > 0) == (layout == 2)
    return p


def run(p, w):
    F, gap = p.forward()
    out = {"F": F, "gap": gap, "fields": [p.field(c) for c in range(6)], "dft": p.dft(),
           "maps": [p.index_map(q) for q in range(4)], "p": p}
    p.adjoint()
    out["adft"], out["grad"] = p.dft(True), p.gradient()
    return out


CASES = ([(parity.test_paired_shell_paths, (s,)) for s in ("tfsf_odd", "tfsf_even", "dipole_shell_odd", "dipole_shell_even", "per_sample")] +
         [(parity.test_paired_design_paths, (c,)) for c in ("gap_odd", "gap_even", "tfsf_in_design_odd", "tfsf_in_design_even",
                                                            "poles8", "no_poles", "per_sample")] +
         [(parity.test_per_sample_density, (32, 52, 1))] + [(parity.test_paper_workload_reduced, (m,)) for m in ("Si", "Au")])


@pytest.mark.parametrize("test,args", CASES, ids=["-".join((t.__name__[5:],) + tuple(map(str, a))) for t, a in CASES])
def test_parity_cases_with_the_interior_kernel(gpu, monkeypatch, test, args):  # noqa: F811
    ran = []

    def run_gpu(lib, w, adjoint=True, rho=None):
        p = problem(lib, w, 2)
        ran.append(p)
        return run(p, w)

    monkeypatch.setattr(parity, "run_gpu", run_gpu)
    test(gpu, *args)
    assert ran


@pytest.mark.parametrize("layout", [1, 2])
@pytest.mark.parametrize("prec", [32, 64])
def test_paper_mode(gpu, prec, layout):  # noqa: F811
    w = _case(prec)
    Fo, go0, go1 = _oracle(w)
    p = problem(gpu, w, layout)
    for interval in (170, 33, 1):                      # 1200 = 7 x 170 + 10: a short last segment; odd starts; every step
        F = p.paper_forward(checkpoint_steps=interval)
        assert abs(F - Fo) <= TOL[prec] * abs(Fo)
        assert rel(p.paper_gradient(pole_pairing=0), go0) <= TOL[prec]
        assert rel(p.paper_gradient(pole_pairing=1), go1) <= TOL[prec]
    p.close()


@pytest.mark.parametrize("interval", [5, 16, 17, 33, 64, 171])
def test_paper_mode_intervals(gpu, interval):  # noqa: F811
    p = problem(gpu, _case(64, steps=311), 2)
    F = p.paper_forward(checkpoint_steps=32)
    g = p.paper_gradient(pole_pairing=1)
    assert p.paper_forward(checkpoint_steps=interval) == F
    assert rel(p.paper_gradient(pole_pairing=1), g) <= 1e-12
    p.close()


# fields, DFTs and gradient of the same handle as it changes layout: the second buffers are stale when it comes back to them
@pytest.mark.parametrize("prec", [32, 64])
def test_layout_changes_between_runs(gpu, prec):  # noqa: F811
    w = _case(prec, steps=421)
    o = run_oracle(w)
    p = gpu.problem(w)
    for layout in (2, 1, 2, 0):
        p.set_step_layout(layout)
        compare(run(p, w), o, prec)
    p.close()


@pytest.mark.parametrize("first,second", [(1, 2), (2, 1)])
def test_layout_changes_between_paper_passes(gpu, first, second):  # noqa: F811
    w = _case(64, steps=311)
    p = problem(gpu, w, first)
    F = p.paper_forward(checkpoint_steps=33)
    g = p.paper_gradient(pole_pairing=1)
    p.set_step_layout(second)
    assert rel(p.paper_gradient(pole_pairing=1), g) <= 1e-12      # the first layout's checkpoints, odd segment starts
    assert abs(p.paper_forward(checkpoint_steps=33) - F) <= 1e-12 * abs(F)
    assert rel(p.paper_gradient(pole_pairing=1), g) <= 1e-12
    assert np.isfinite(p.forward()[0])                            # a plain run after them
    p.close()


# x rows of no multiple of 32 bytes: the box starts on 16 bytes where that keeps a mostly full last tile column
@pytest.mark.parametrize("prec,nx,cpml_x,box_x", [(32, 76, 8, (12, 68)), (32, 68, 8, (16, 48)), (64, 90, 12, (14, 78)),
                                                   (64, 78, 5, (8, 72))])
def test_box_start_of_odd_rows(gpu, prec, nx, cpml_x, box_x):  # noqa: F811
    d = base_desc(nx, 42, 37, n_steps=420, cpml=(cpml_x, cpml_x, 4, 7, 5, 3), precision=prec, design=(22, 18, 15), gap=(2, 2, 2),
                  lambdas_nm=(500.0, 650.0), src_kind=1, src_pos=(cpml_x + 3, 0, 0))
    w = dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(23, 3), gamma=1e6,
             rho=synth.smooth_rho(synth.box_shape(d["design_box"]), 23, 2.0))
    p = problem(gpu, w, 2)
    assert p.timings()["interior_cells"] == (box_x[1] - box_x[0]) * 30 * 28
    compare(run(p, w), run_oracle(w), prec)
    p.close()
