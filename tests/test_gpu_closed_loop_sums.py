"""The closed loop's control sums over the nodes: partial sums in pairs of floats
are added across the block without losing bits that FP64 holds.

At the corner of two end points of a level-2 grid the control is the sum of
three surpluses whose products are exact; with values 1, 2^-25 and 2^-52 the
sum needs 53 bits, which FP64 has and a pair of floats has not, so every
arithmetic must give it exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu
LO, HI = synth.box(6)


@pytest.mark.parametrize("mode", [sg.EVAL_FP64, sg.EVAL_DF32], ids=["fp64", "df32"])
@pytest.mark.parametrize("n", [1, 305, 609])      # one, two and four trajectories per block
def test_partial_controls_keep_53_bits(n, mode):
    g = sg.Grid(6, 2, LO, HI)
    x = g.coords.cpu().numpy()
    end = np.abs(x - HI) < 1e-12
    f = 1.0 + 2.0 ** -25 * end[:, 0] + 2.0 ** -52 * end[:, 1]
    S = sg.Surplus(g, torch.as_tensor(np.repeat(f[:, None], 3, 1), device="cuda"))
    corner = int(np.flatnonzero(end[:, 0] & end[:, 1])[0])
    out = sg.simulate_closed_loop(sg.problem_from(synth.attitude_params(0)), S,
                                  g.coords[corner].repeat(n, 1).contiguous(), 1, 0.01, mode=mode,
                                  keep_trajectory=True)
    u = out["ctrl"][:, 0].cpu().numpy()
    assert np.all(u == 1.0 + 2.0 ** -25 + 2.0 ** -52)


@pytest.mark.parametrize("mode", [sg.EVAL_FP64, sg.EVAL_DF32], ids=["fp64", "df32"])
@pytest.mark.parametrize("level", [4, 5])
def test_block_forms_where_shared_memory_is_fullest(level, mode):
    """Level 4 keeps its nodes in shared memory beside one, two or four trajectories'
    tables (48 KB with the static part), level 5 reads them from global memory:
    every form launches and gives the same bits."""
    g = sg.Grid(6, level, LO, HI)
    v = -(g.coords[:, :3] + 2.0 * g.coords[:, 3:])
    S = sg.Surplus(g, v.contiguous())
    prob = sg.problem_from(synth.attitude_params(1))
    x0 = torch.as_tensor(synth.uniform_queries(700, LO, HI, seed=12), device="cuda")
    full = sg.simulate_closed_loop(prob, S, x0, 3, 0.01, mode=mode)
    for n in (2, 400):
        part = sg.simulate_closed_loop(prob, S, x0[:n].contiguous(), 3, 0.01, mode=mode)
        for key in ("xT", "cost"):
            assert torch.equal(part[key], full[key][:n]), (n, key)
