"""The closed loop's sines and cosines over their branches: the polynomials, the
two-part reduction by one and two quarter turns of either sign, and the library
beyond 3.875; attitudes far outside the usual box, against the oracle's step
(1e-10, the closed loop's stated tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from oracle import closed_loop as ocl  # noqa: E402
from oracle import grid as ogrid  # noqa: E402
from oracle import interp as ointerp  # noqa: E402
from oracle import problems as oprob  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu

ANGLES = [0.2, 0.7853, 0.7855, 1.3, 1.7, 2.3, 2.4, 3.0, 3.2, 3.87, 3.88, 4.3]


@pytest.mark.parametrize("mode", [sg.EVAL_FP64, sg.EVAL_DF32], ids=["fp64", "df32"])
def test_quarter_turns_match_oracle(mode):
    lo, hi = synth.box(6, half=5.0)
    g, og = sg.Grid(6, 1, lo, hi), ogrid.Grid(6, 1, lo, hi)
    f = np.random.default_rng(71).standard_normal((og.M, 3))
    S = sg.Surplus(g, torch.as_tensor(f, device="cuda"))
    w = ointerp.surpluses(og, f)
    s = [a * sgn for a in ANGLES for sgn in (1.0, -1.0)]
    n = len(s)
    X0 = np.zeros((n, 6))
    X0[:, 0] = s
    X0[:, 1] = np.roll(s, 5)        # (cos theta is at least 0.12 at these angles)
    X0[:, 2] = np.roll(s, 11)
    X0[:, 3:] = np.random.default_rng(72).uniform(-0.5, 0.5, (n, 3))
    params = synth.attitude_params(0)
    out = sg.simulate_closed_loop(sg.problem_from(params), S, torch.as_tensor(X0, device="cuda"), 2, 0.01, mode=mode,
                                  keep_trajectory=True)
    pr = oprob.make(params)
    for i in range(n):
        xs, us, z = ocl.simulate(pr, og, w, X0[i], 2, 0.01)
        assert np.max(np.abs(out["ctrl"][i].cpu().numpy() - us)) <= 1e-10 * np.max(np.abs(us)), X0[i]
        assert np.max(np.abs(out["traj"][i].cpu().numpy() - xs)) <= 1e-10 * np.max(np.abs(xs)), X0[i]
        assert abs(out["cost"][i].item() - z) <= 1e-10 * z, X0[i]
