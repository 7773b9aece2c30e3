"""FP64 rows of the 1-D basis where a difference to a grid point is below the
normal range, and far outside the box: finite wherever the barycentric form in
correctly rounded arithmetic is, and next to a grid point the value there."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu

# (below 2^-1024 the reciprocal itself is infinite)
TINY = [6e-309, 1e-308, 2e-308, -1e-308, 3e-308, 1e-300, 1e-290]


def _cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _surplus(d, L, k=3):
    g = sg.Grid(d, L, np.zeros(d), np.ones(d))
    return sg.Surplus(g, _cuda(np.random.default_rng(60 + L).standard_normal((g.M, k))))


@pytest.mark.parametrize("repeat", [1, 900])      # both launch forms
@pytest.mark.parametrize("d,L", [(1, 1), (2, 3), (1, 5), (6, 2), (2, 6)])
def test_next_to_a_grid_point(d, L, repeat):
    S = _surplus(d, L)
    q = np.full((len(TINY) + 1, d), 0.3)
    q[0, 0], q[1:, 0] = 0.0, TINY
    u = sg.eval_feedback(S, _cuda(np.tile(q, (repeat, 1)))).cpu().numpy()
    # the interpolant's slope is at most a few hundred, so the values agree to rounding
    assert np.max(np.abs(u - u[0])) <= 1e-12 * np.max(np.abs(u[0]))


@pytest.mark.parametrize("repeat", [1, 1700])
def test_far_outside_the_box(repeat):
    S = _surplus(1, 5)
    q = np.tile(np.array([[4.0], [100.0], [-3.0], [0.25]]), (repeat, 1))
    assert np.all(np.isfinite(sg.eval_feedback(S, _cuda(q)).cpu().numpy()))


def test_closed_loop_next_to_a_grid_point():
    S = _surplus(6, 2)
    q = np.full((len(TINY) + 1, 6), 0.3)
    q[0, 0], q[1:, 0] = 0.0, TINY
    o = sg.simulate_closed_loop(sg.problem_from(synth.attitude_params(0)), S, _cuda(q), 1, 0.01,
                                mode=sg.EVAL_FP64, keep_trajectory=True)
    u = o["ctrl"].cpu().numpy()[:, 0]
    assert np.max(np.abs(u - u[0])) <= 1e-12 * np.max(np.abs(u[0]))
