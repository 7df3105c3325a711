"""Paper mode's passes as 16-step graph replays: checkpoint intervals that make a segment start at an odd step, end in
a remainder, or hold no whole graph give the gradient of every other interval (the order of steps does not change;
1e-12 in FP64 leaves room for another contraction of the same operations)."""
import pytest

from parity_util import rel
from test_paper_mode_gpu import _case, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interval", [5, 16, 17, 33, 64, 171])
def test_intervals(lib, interval):  # noqa: F811
    w = _case(64, steps=311)
    p = lib.problem(w)
    F = p.paper_forward(checkpoint_steps=32)
    g = [p.paper_gradient(pole_pairing=q) for q in (0, 1)]
    assert p.paper_forward(checkpoint_steps=interval) == F
    for q in (0, 1):
        assert rel(p.paper_gradient(pole_pairing=q), g[q]) <= 1e-12
    p.close()
