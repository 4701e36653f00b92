"""The captured steps against the level-by-level steps of timing mode 1, bit for
bit, on meshes beyond 2^20 elements (every storage type and time mode, a force,
instants of two of three levels) and with interpolated bounce-back; and there
the state and ghosts that the adjoint's recording leaves, against lbm_step's."""
import functools

import numpy as np
import pytest

from paper_1601_06984_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu
P6 = (W.BC_PERIODIC,) * 6


@functools.lru_cache(maxsize=1)
def mesh(name):
    if name == "two levels":    # 7.7e5 + 8.8e5 elements: only the first instant is beyond
        return W.nested_boxes(3, 7, (96, 96, 96), [((48, 48, 48), (144, 144, 144))], P6)
    if name == "three levels":  # 6.2e5 + 1.8e6 + 2.1e6: all instants are
        return W.nested_boxes(3, 7, (96, 96, 96), [((32, 32, 32), (160, 160, 160)), ((128, 128, 128), (256, 256, 256))], P6)
    return W.config_cylinder_schafer(20)


def sim(name, precision, mode, force=False, tape=0):
    m = mesh(name)
    walls = name == "channel"
    Q = 9 if m.d == 2 else 19
    om = W.omega_coarse_from_finest(1.6, len(m.level_counts())) if mode != 2 else 1.6
    s = lbm.Sim(m, Q, om, precision=precision, time_mode=mode, use_force=force, u_in=(0.05, 0, 0) if walls else (0, 0, 0),
                inlet_profile=int(walls), bouzidi=walls, adjoint_tape=tape)
    if walls:
        e, d = s.obstacle_links()
        s.set_link_q(W.wall_distance_ball(m, e, d, (40.0, 40.0), 10.0, 9))
    rng = np.random.default_rng(1601)
    u = 0.03 * rng.standard_normal((m.n, m.d))
    s.init(1.0 + 1e-3 * rng.standard_normal(m.n), u)
    if force:
        s.set_force(1e-5 * rng.standard_normal((m.n, m.d)))
    return s


@pytest.mark.parametrize("name,precision,mode,force", [
    ("two levels", 0, 0, False), ("two levels", 0, 1, True), ("two levels", 1, 0, True), ("two levels", 1, 2, False),
    ("two levels", 2, 0, True), ("two levels", 2, 2, False), ("three levels", 1, 0, False), ("three levels", 2, 1, False),
    ("three levels", 2, 0, False), ("channel", 0, 0, False), ("channel", 0, 1, False), ("channel", 1, 0, False)])
def test_captured_steps_equal_level_by_level(name, precision, mode, force):
    out = []
    for timing in (0, 1):
        s = sim(name, precision, mode, force)
        s.timing_enable(timing)
        for n in (1, 2):  # from both parities
            s.step(n)
        out.append((s.get_state(), s.ghosts()[1]))
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("tape", [1, 2])
@pytest.mark.parametrize("name,precision,mode", [("two levels", 1, 0), ("two levels", 1, 1), ("three levels", 1, 0)])
def test_adjoint_leaves_the_state_and_ghosts_of_the_steps(name, precision, mode, tape):
    out = []
    for adjoint in (False, True):
        s = sim(name, precision, mode, tape=tape)
        s.step(1)
        s.adjoint(2, 1, 0, want_force=False) if adjoint else s.step(2)
        out.append((s.get_state(), s.ghosts()[1]))
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
