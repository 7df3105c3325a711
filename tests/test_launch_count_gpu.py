"""The launch count that fdtd_timings gives against the kernels the device ran (torch's profiler records them, those of
graph replays too): plain runs with the E phase in one launch and in two, with an interior kernel, and paper mode, whose
passes mix graph replays with single steps."""
import pytest

import synth
from synth import base_desc, vacuum
from test_paper_mode_gpu import _case, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def recording(lib):  # noqa: F811
    """The profiler's first session starts its recorder and may miss what runs in it."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):
        torch.ones(8, device="cuda").sum().item()


def counted(p, call):
    """(kernels of this library that ran during the call, launches the handle reports for it)"""
    from torch.profiler import ProfilerActivity, profile
    before = p.timings()["launches"]
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
    names = [e.name for e in prof.events() if "fdtd::" in e.name or "_kernel" in e.name]
    if not names:
        pytest.skip("the profiler records no kernels here")
    return len(names), p.timings()["launches"] - before


# E phase in one launch; in two (72^3: columns of several planes); the interior kernel
@pytest.mark.parametrize("n,layout", [(48, 0), (72, 1), (72, 2)])
@pytest.mark.parametrize("steps", [48, 53])
def test_plain_runs(lib, n, layout, steps):  # noqa: F811
    d = base_desc(n, n, n, n_steps=steps, cpml=6, design=(16, 16, 16), gap=(2, 2, 2))
    d["src_t0"], d["src_fwhm_hz"], d["adj_tau"] = 20 * d["courant"] * d["dx"] / synth.C0, 2e15, 1.5e-16
    p = lib.problem(dict(desc=d, bg=vacuum(), m1=vacuum(), m2=synth.drude_lorentz_metal(3, 1), gamma=0.0,
                         rho=synth.uniform_rho((16, 16, 16), 3)))
    p.set_step_layout(layout)
    p.forward()                                        # graphs built
    ran, said = counted(p, p.forward)
    assert ran == said
    ran, said = counted(p, p.adjoint)
    assert ran == said
    p.close()


@pytest.mark.parametrize("interval", [16, 33, 160])
def test_paper_mode(lib, interval):  # noqa: F811
    p = lib.problem(_case(64, steps=311))
    p.paper_forward(checkpoint_steps=interval)
    for call in (lambda: p.paper_forward(checkpoint_steps=interval), p.paper_gradient):
        ran, said = counted(p, call)
        assert ran == said
    p.close()
