"""The captured steps (levels batched by instant, launches shared and chained)
against the level-by-level steps of timing mode 1, bit for bit, on meshes on
both sides of every line of the dispatch; and the state and ghosts that the
adjoint's tape leaves, against lbm_step's."""
import numpy as np
import pytest

from paper_1601_06984_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1601_06984_gb300 import build, lbm as L
    build.build()
    return L


def deep2d(levels):
    """Nested 2D boxes, `levels` deep: seven exceed the levels one launch takes."""
    boxes, lo, hi = [], (0, 0), (32, 32)
    for _ in range(levels - 1):
        w = [b - a for a, b in zip(lo, hi)]
        lo, hi = tuple(2 * (a + n // 4) for a, n in zip(lo, w)), tuple(2 * (b - n // 4) for b, n in zip(hi, w))
        boxes.append((lo, hi))
    return W.nested_boxes(2, 5, (32, 32), boxes, (W.BC_PERIODIC,) * 4)


MESHES = {
    "one level": lambda: W.uniform(2, 5, (32, 24), (W.BC_PERIODIC,) * 4),
    "tiny": W.config_tgv2d,                              # below the FP64 chain's line
    "ragged": lambda: W.nested_boxes(3, 6, (37, 22, 19), [((18, 10, 8), (56, 34, 30))], (W.BC_PERIODIC,) * 6),
    "6 levels": lambda: deep2d(6),
    "7 levels": lambda: deep2d(7),                       # the recursion's launches
    "sphere": W.config_sphere_5level_small,              # outlet, inlet, obstacle
    # 1.7e6 elements: beyond the chain's line
    "large": lambda: W.nested_boxes(3, 7, (96, 96, 96), [((48, 48, 48), (144, 144, 144))], (W.BC_PERIODIC,) * 6),
}
CASES = [("one level", 9, 1, 0), ("tiny", 9, 0, 0), ("tiny", 9, 0, 2), ("tiny", 9, 2, 1), ("ragged", 19, 0, 0),
         ("ragged", 19, 1, 1), ("ragged", 27, 1, 0), ("ragged", 27, 0, 1), ("ragged", 19, 2, 1), ("6 levels", 9, 0, 0),
         ("6 levels", 9, 1, 1), ("7 levels", 9, 0, 0), ("7 levels", 9, 1, 1), ("sphere", 19, 0, 1), ("sphere", 27, 1, 1),
         ("sphere", 19, 2, 0), ("large", 19, 1, 0), ("large", 19, 2, 1)]


@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("name,Q,precision,mode", CASES)
def test_captured_steps_equal_level_by_level(lbm, name, Q, precision, mode, force):
    if name == "large" and force:
        pytest.skip("the size matters here, and the mesh is slow to build")
    m = MESHES[name]()
    inlet = name == "sphere"
    om = W.omega_coarse_from_finest(1.6, len(m.level_counts()))
    sims = []
    for timing in (0, 1):
        s = lbm.Sim(m, Q, om, precision=precision, time_mode=mode, use_force=force, outlet=1,
                    u_in=(0.04, 0, 0) if inlet else (0, 0, 0))
        u0 = (0.04, 0.0, 0.0)[: m.d]
        s.init(*W.uniform_fields(m, 1.0, u0), W.pdf_perturbation(m, Q, 1e-3) if m.n < 500_000 else None)
        if force:
            s.set_force(W.gaussian_force(m, 1e-4))
        s.timing_enable(timing)
        for n in (1, 4, 1):  # one-step and two-step graphs from both parities
            s.step(n)
        sims.append(s)
    a, b = sims
    assert np.array_equal(a.get_state(), b.get_state())
    assert np.array_equal(a.ghosts()[1], b.ghosts()[1])


@pytest.mark.parametrize("tape", [1, 2])
@pytest.mark.parametrize("n,K", [(1, 1), (5, 2), (3, 5)])
@pytest.mark.parametrize("name,mode", [("tiny", 0), ("tiny", 1), ("sphere", 0), ("sphere", 1)])
def test_adjoint_leaves_the_state_and_ghosts_of_the_steps(lbm, name, mode, n, K, tape):
    m = MESHES[name]()
    Q = 9 if m.d == 2 else 19
    out = []
    for adjoint in (False, True):
        s = lbm.Sim(m, Q, W.omega_coarse_from_finest(1.6, len(m.level_counts())), time_mode=mode, outlet=1,
                    u_in=(0.04, 0, 0) if name == "sphere" else (0, 0, 0), adjoint_tape=tape)
        s.init(*W.uniform_fields(m, 1.0, (0.04, 0.0, 0.0)[: m.d]), W.pdf_perturbation(m, Q, 1e-3))
        s.fill_ghosts()
        s.step(1)
        s.adjoint(n, K, 0) if adjoint else s.step(n)
        out.append([s.get_state(), s.ghosts()[1]])
        s.step(2)
        out[-1] += [s.get_state(), s.ghosts()[1]]
    for a, b in zip(*out):
        assert np.array_equal(a, b)
