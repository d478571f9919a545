"""The bound of the network policies' estimate: the host arithmetic alone (the kernels that use it are compared with
the defined logits on the GPU). Two logits of the same weights can never differ, so the estimate, which is zero then,
has to decide: a network whose last layer starts at zero computed its defined logits in every step otherwise. And the bound
has to count every rounding of the kernels' orders, or it is not the one that was derived."""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_13062_b200 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
UNITS = {inputs.POLICY_MLP: 16, inputs.POLICY_MLP32: 32, inputs.POLICY_MLP64: 64, inputs.POLICY_MLP_DEEP: 16}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("bound") / "policy_bound")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-O1", os.path.join(ROOT, "tests", "policy_bound_program.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def bound(program):
    exe = program

    def call(kind, w):
        h = UNITS[kind]
        args = [exe, str(h), str(int(kind == inputs.POLICY_MLP_DEEP)), str(h)]
        out = subprocess.run(args, input=w.astype(np.float32).tobytes(), check=True, capture_output=True).stdout
        return [float(v) for v in out.split()]
    return call


def last_layer(kind, w):
    h = UNITS[kind]
    last = w[w.size - 2 * h - 2:]
    return last[:2 * h].reshape(2, h), last[2 * h:]


@pytest.mark.parametrize("kind", list(UNITS))
def test_logits_of_the_same_weights(bound, kind):
    w = inputs.policy_weights(kind, 11)
    rows, bias = last_layer(kind, w)
    assert bound(kind, w)[1] > 0.0
    rows[1], bias[1] = rows[0], bias[0]
    base, decides, step = bound(kind, w)
    assert base == 0.0 and step == 0.0 and decides < 0.0        # |0| > bound, and never pushes right
    rows[:], bias[:] = 0.0, 0.0
    rows[1, 3] = -0.0                                            # the sign of a zero moves no logit away from the other
    base, decides, step = bound(kind, w)
    assert base == 0.0 and step == 0.0 and decides < 0.0


@pytest.mark.parametrize("kind", list(UNITS))
def test_logits_one_bit_apart_are_not_the_same(bound, kind):
    for move in range(3):
        w = inputs.policy_weights(kind, 11)
        rows, bias = last_layer(kind, w)
        rows[1], bias[1] = rows[0], bias[0]
        target = (rows[1], bias[1:], rows[0])[move]
        target[-1] = np.nextafter(target[-1], np.float32(9.0))
        assert bound(kind, w)[1] > 0.0


@pytest.mark.parametrize("value", [np.float32(1e30), np.float32(np.inf), np.float32(np.nan)])
@pytest.mark.parametrize("kind", list(UNITS))
def test_weights_that_may_overflow_never_decide(bound, kind, value):
    for same in (False, True):
        w = inputs.policy_weights(kind, 11)
        rows, bias = last_layer(kind, w)
        rows[:, 2] = value
        if same:
            rows[1], bias[1] = rows[0], bias[0]
        assert bound(kind, w)[1] == np.inf


class Rounded:
    """A sum that counts the roundings each term of it has gone through: `most` of the terms', None without a term."""

    def __init__(self, most=None):
        self.most = most

    def plus(self, *others):
        """One operation, a multiply-add or a sum: whatever goes into it is rounded once more."""
        terms = [o.most for o in (self, *others) if o.most is not None]
        return Rounded(max(terms) + 1)


TERM = Rounded(0)   # w * h before the operation that rounds it, or the base, or 0


def spread_over_lanes(units, lanes):
    """The order of lanes_action (rollout_lanes.cuh), every lane alike."""
    mine = units // lanes
    if lanes <= 2:
        half = TERM.plus()                              # mul2
        for _ in range(1, mine // 2):
            half = half.plus(TERM)                      # fma2
        part = half.plus(half)                          # low + high half
    else:
        part = TERM
        for _ in range(mine):
            part = part.plus(TERM)                      # fma from 0
    while lanes > 1:
        part, lanes = part.plus(part), lanes // 2       # shuffles
    return part.plus(TERM)                              # the base


def paired_layout(units, deep):
    """The orders of screen_estimate and screen_estimate_two (policy_screen.cuh)."""
    est = TERM
    for _ in range(units if deep else units // 2):
        est = est.plus(TERM)
    return est if deep else est.plus(TERM)


# the instances of the lane-split kernel whose weights are the lanes' own (launch_lanes_g), as (policy, lanes)
SPREAD = [(kind, 4) for kind in UNITS] + [(inputs.POLICY_MLP, 1), (inputs.POLICY_MLP, 2), (inputs.POLICY_MLP32, 2)] + \
    [(kind, 8) for kind in UNITS]


@pytest.mark.parametrize("kind,lanes", SPREAD + [(kind, 0) for kind in UNITS])
def test_no_term_goes_through_more_roundings_than_the_bound_counts(program, kind, lanes):
    deep = kind == inputs.POLICY_MLP_DEEP
    args = [program, "rounds", str(UNITS[kind]), str(int(deep)), str(lanes)]
    stated = int(subprocess.run(args, check=True, capture_output=True).stdout)
    needed = (spread_over_lanes(UNITS[kind], lanes) if lanes else paired_layout(UNITS[kind], deep)).most
    assert stated >= needed
