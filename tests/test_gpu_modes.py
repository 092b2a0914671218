"""Which elimination a context takes follows from the states of its options, not from the order in
which they were set; putting an option back puts its effect back."""
import numpy as np
import pytest

from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _same(a, b):
    return np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
def test_option_orders(prec):
    p = api.Params(14, 3, U=4.0, T=0.3, delta=0.4, prec=prec)
    phi = inputs.random_phi(1, p.N, 1.0)

    def after(*calls):
        with api.Context(p) as c:
            for name, arg in calls:
                getattr(c, name)(arg)
            return c.blocks(phi)

    new, dense = after(), after(("set_pivoting", "partial"))
    assert not _same(new, dense)
    # back to what a new context takes
    for calls in ([("set_pivoting", "auto")],
                  [("set_pivoting", "partial"), ("set_pivoting", "auto")],
                  [("set_pivoting", "none"), ("set_pivoting", "auto")],
                  [("set_pivoting", "partial"), ("set_pivoting", "none")],
                  [("set_panel_precision", "fp32")],
                  [("set_panel_precision", "fp64"), ("set_panel_precision", "fp32")],
                  [("set_panel_precision", "fp64"), ("set_pivoting", "none"),
                   ("set_panel_precision", "fp32")],
                  [("profile", True), ("profile", False)]):
        assert _same(after(*calls), new), calls
    # float64 panels: the dense elimination, whichever way the pivoting was set before or after
    panels = after(("set_panel_precision", "fp64"))
    assert not _same(panels, new) and not _same(panels, dense)
    assert _same(after(("set_pivoting", "partial"), ("set_panel_precision", "fp64")), panels)
    assert _same(after(("set_panel_precision", "fp64"), ("set_pivoting", "auto")), panels)
    a = after(("set_panel_precision", "fp64"), ("set_pivoting", "none"))
    b = after(("set_pivoting", "none"), ("set_panel_precision", "fp64"))
    assert _same(a, b) and not _same(a, new)


def test_auto_below_the_line_pivots():
    """pi T < 0.03: 'auto' after 'none' is a new context's pivoted dense elimination again."""
    p = api.Params(14, 4, U=4.0, T=0.008, delta=0.4, prec="fp64")
    phi = inputs.random_phi(2, p.N, 1.0)
    with api.Context(p) as c:
        new = c.blocks(phi)
        c.set_pivoting("none")
        none = c.blocks(phi)
        c.set_pivoting("auto")
        assert _same(c.blocks(phi), new) and not _same(none, new)


def test_profile_takes_any_truth_value():
    p = api.Params(8, 2, U=4.0, T=0.3, delta=0.4, prec="fp32")
    phi = inputs.random_phi(4, p.N, 1.0)
    with api.Context(p) as c:
        for enable, dense, nested in ((None, 0, 0), ("", 0, 0), ("on", 1, 0), (True, 1, 0), (2, 0, 1),
                                      (5, 1, 0), (0, 0, 0)):
            c.profile(enable)
            c.blocks(phi)
            prof = c.profile_read()
            assert (prof["panel"][1] > 0) == bool(dense), enable
            assert (prof["nest_up"][1] > 0) == bool(nested), enable


def test_environment_switch_counts_at_creation(monkeypatch):
    p = api.Params(14, 3, U=4.0, T=0.3, delta=0.4, prec="bf16x3")
    phi = inputs.random_phi(3, p.N, 1.0)
    with api.Context(p) as c:
        new = c.blocks(phi)
        monkeypatch.setenv("SCA_REFINE_LOWER", "1")
        c.set_pivoting("none")
        assert _same(c.blocks(phi), new)
    with api.Context(p) as c:
        monkeypatch.delenv("SCA_REFINE_LOWER")
        switched = c.blocks(phi)
        c.set_pivoting("auto")
        assert _same(c.blocks(phi), switched) and not _same(switched, new)
