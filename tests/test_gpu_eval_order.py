"""An FP64 evaluation's result at a query is the same to the last bit whatever
the number of queries in the call: the sum over the nodes has one order in every
launch form.  Checked across the counts at which the form changes, and for
evaluations that a server merges."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from paper_1507_04769_gb300 import serving, sg  # noqa: E402

pytestmark = pytest.mark.gpu

COUNTS = [1, 5, 31, 152, 153, 304, 305, 608, 609, 1216, 1217, 1824, 1825, 2432, 2433, 4864, 4865, 9728, 9729, 14593, 19457]


@pytest.mark.parametrize("d,L,k", [(6, 4, 3), (6, 5, 3), (6, 2, 7), (8, 3, 6), (1, 6, 2), (5, 0, 1), (2, 5, 16)])
def test_rows_do_not_depend_on_the_number_of_queries(d, L, k):
    lo, hi = synth.box(d)
    g = sg.Grid(d, L, lo, hi)
    S = sg.Surplus(g, torch.as_tensor(np.random.default_rng(90 + d).standard_normal((g.M, k)), device="cuda"))
    xq = torch.as_tensor(synth.mixed_queries(20001, lo, hi, seed=91), device="cuda")
    xq[:min(g.M, 40)] = g.coords[:40]
    xq[40:60] *= 1.1                       # outside the box
    full = sg.eval_feedback(S, xq)
    assert bool(torch.isfinite(full).all())
    for n in COUNTS:
        assert torch.equal(sg.eval_feedback(S, xq[:n].contiguous()), full[:n]), n


def test_fp64_evaluations_served_in_a_mix_match_solo():
    server = serving.Server(slots=2, pool_slots=256, eval_mode=sg.EVAL_FP64)
    keys = [(2, 20.0)]
    counts = server.warm(levels=(2,), model_keys=keys)
    reqs = serving.make_requests(16, rate=1e4, node_counts=counts, seed=6, levels=(2,), horizons=(20.0,),
                                 mix=(0, 1, 0), max_queries=5000, max_traj=16, nsteps=50, model_keys=keys)
    server.start()
    done = serving.replay(server, reqs, realtime=False)
    assert len(done) == len(reqs) and any(r.batch_size > 1 for r in done)
    m = server.models[keys[0]]
    for r in done:
        solo = sg.eval_feedback(m.surplus, torch.as_tensor(r.x, device="cuda"), mode=sg.EVAL_FP64)
        assert np.array_equal(r.result["u"], solo.cpu().numpy()), r.rid
