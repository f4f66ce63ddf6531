"""The autotuner's search over launch shapes returns the settings that it timed: applied to new
operators they give the state behind the returned time.  On the CPU, with stand-ins for the
operators whose automatic shapes are no setting of any knob."""
import itertools

import pytest

from paper_2112_15562_gb300 import autotune
from paper_2112_15562_gb300._lib import GJ_TUNE_AUTO, GJError


class FakeOp:
    """The launch shapes as gj_op_tune keeps them; None: the library's own, pass by pass."""

    def __init__(self):
        self.state = {"P_row": None, "C_col": None, "L_grp": None, "radix_order": 0}

    def tiles(self):  # of both fields' launches
        return {"P_row": 8, "C_col": 4, "L_grp": 4, "radix_order": self.state["radix_order"]}

    def tune(self, P_row=0, C_col=0, L_grp=0, radix_order=-1):
        for k, v in (("P_row", P_row), ("C_col", C_col), ("L_grp", L_grp)):
            if v == 16 and k == "C_col":
                raise GJError(-1, "too large")
            if v > 0 or v == GJ_TUNE_AUTO:
                self.state[k] = None if v == GJ_TUNE_AUTO else v
        if radix_order >= 0:
            self.state["radix_order"] = radix_order


COSTS = [{}, {"P_row": {2: -1.0}}, {"P_row": {1: -1.0, 2: -2.0}, "L_grp": {8: -3.0}}, {"radix_order": {1: -2.0}},
         {"C_col": {1: -1.0, 16: -9.0}, "radix_order": {2: -1.0}}]


# what a shape pinned to the reported one costs against the library's own choice for every pass
@pytest.mark.parametrize("gains,pinned", list(itertools.product(COSTS, (-0.5, 0.0, 0.5))))
def test_the_returned_settings_are_the_timed_ones(monkeypatch, gains, pinned):
    def cost(op):
        t = 10.0
        for k, v in op.state.items():
            t += gains.get(k, {}).get(v, 0.0)
            if k != "radix_order" and v == op.tiles()[k]:
                t += pinned
        return t

    monkeypatch.setattr(autotune, "_time_ops", lambda ops, reps: max(cost(op) for op in ops))
    ops = [FakeOp(), FakeOp()]
    settings, time = autotune._refine(ops, 2, cost(FakeOp()))
    new = FakeOp()
    if settings:
        new.tune(**settings)
    assert cost(new) == pytest.approx(time)
    assert all(op.state == new.state for op in ops)
    assert all(v in autotune.KNOBS[k] for k, v in settings.items())
