"""FP32 eliminations with pivots near the largest float: the cost of a
linear-quadratic problem scaled by 2^e scales the costates and nothing else, and
takes the staircase's and the closing system's pivots (the terminal weight is
2^e) out of the range of the reciprocal's short form.  lambda(0) / 2^e agrees
with the unscaled solve's within the 1e-6 stated for solves stopped at 1e-8."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu
LO, HI = synth.box(6)


def _solve(e, N):
    p = synth.lq_params(0)
    s = 2.0 ** e
    p.Q, p.R, p.QT = p.Q * s, p.R * s, p.QT * s
    X = torch.as_tensor(synth.uniform_queries(40, LO, HI, seed=5), device="cuda")
    r = sg.solve_bvps(sg.problem_from(p), X, 10.0, N, tol=1e-8 * s, precision=sg.PREC_MIXED)
    assert torch.all(r["status"] == sg.CONVERGED) and int(r["iters"].max()) <= 2
    return r["lambda0"].cpu().numpy() / s


@pytest.mark.parametrize("e,N", [(100, 16), (125, 16), (125, 40), (126, 40)])
def test_scaled_cost_scales_the_costates(e, N):
    ref = _solve(0, N)
    assert np.max(np.abs(_solve(e, N) - ref)) <= 1e-6 * np.max(np.abs(ref))
