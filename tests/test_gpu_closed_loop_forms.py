"""The closed loop over its launch forms: one, two and four trajectories per
block give bitwise the same trajectory, every level's
tables and the other plant families match the oracle within the
closed loop's stated 1e-10, from states inside the box, at nodes and with
angles beyond pi/4."""
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
LO, HI = synth.box(6)


def _values(x):
    return -(x[:, :3] + 2.0 * x[:, 3:]) - 0.1 * np.sin(x[:, :3] * x[:, 3:])


def _rel(a, b):
    return np.max(np.abs(np.asarray(a) - b)) / max(np.max(np.abs(b)), 1e-300)


@pytest.mark.parametrize("mode", [sg.EVAL_FP64, sg.EVAL_DF32], ids=["fp64", "df32"])
@pytest.mark.parametrize("level", [0, 1, 2, 3, 4, 5])
def test_levels_match_oracle(level, mode):
    params = synth.attitude_params(0)
    g = sg.Grid(6, level, LO, HI)
    og = ogrid.Grid(6, level, LO, HI)
    S = sg.Surplus(g, torch.as_tensor(_values(g.coords.cpu().numpy()), device="cuda"))
    w = ointerp.surpluses(og, _values(og.x))
    X0 = np.concatenate([synth.uniform_queries(2, LO, HI, seed=level), og.x[:min(3, og.M)],
                         np.array([[0.9, -0.1, 0.05, 0.0, 0.1, 0.0]])])
    nsteps = 6
    out = sg.simulate_closed_loop(sg.problem_from(params), S, torch.as_tensor(X0, device="cuda"), nsteps, 0.01,
                                  mode=mode, keep_trajectory=True)
    pr = oprob.make(params)
    for i in range(X0.shape[0]):
        if level == 5 and i == X0.shape[0] - 1:
            # 7 % outside the box a Lagrange polynomial of degree 32 grows to
            # T_32(1.146) = 1e7, so FP64 rounding of the data alone is 1e-9 there
            continue
        xs, us, z = ocl.simulate(pr, og, w, X0[i], nsteps, 0.01)
        scale = max(np.max(np.abs(us)), 1e-3)
        assert np.max(np.abs(out["ctrl"][i].cpu().numpy() - us)) <= 1e-10 * scale, i
        assert _rel(out["traj"][i].cpu().numpy(), xs) <= 1e-10 or np.max(np.abs(xs)) == 0.0
        assert abs(out["cost"][i].item() - z) <= 1e-10 * max(z, 1e-12)


@pytest.mark.parametrize("mode", [sg.EVAL_FP64, sg.EVAL_DF32], ids=["fp64", "df32"])
def test_trajectories_per_block_bitwise(mode):
    g = sg.Grid(6, 3, LO, HI)
    S = sg.Surplus(g, torch.as_tensor(_values(g.coords.cpu().numpy()), device="cuda"))
    prob = sg.problem_from(synth.attitude_params(1))
    x0 = torch.as_tensor(synth.uniform_queries(611, LO, HI, seed=9), device="cuda")
    full = sg.simulate_closed_loop(prob, S, x0, 20, 0.01, mode=mode, keep_trajectory=True)
    for n in (1, 3, 304, 305, 608):
        part = sg.simulate_closed_loop(prob, S, x0[:n].contiguous(), 20, 0.01, mode=mode, keep_trajectory=True)
        for key in ("xT", "cost", "traj", "ctrl"):
            assert torch.equal(part[key], full[key][:n]), (n, key)


def test_linear_plant_matches_oracle():
    params = synth.lq_params(0)
    g, og = sg.Grid(6, 2, LO, HI), ogrid.Grid(6, 2, LO, HI)
    S = sg.Surplus(g, torch.as_tensor(_values(g.coords.cpu().numpy()), device="cuda"))
    w = ointerp.surpluses(og, _values(og.x))
    X0 = synth.uniform_queries(3, LO, HI, seed=5)
    out = sg.simulate_closed_loop(sg.problem_from(params), S, torch.as_tensor(X0, device="cuda"), 10, 0.01,
                                  mode=sg.EVAL_FP64)
    for i in range(3):
        xs, _, z = ocl.simulate(oprob.make(params), og, w, X0[i], 10, 0.01)
        assert _rel(out["xT"][i].cpu().numpy(), xs[-1]) <= 1e-10
        assert abs(out["cost"][i].item() - z) <= 1e-10 * z
