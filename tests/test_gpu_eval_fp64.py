"""The FP64 evaluation at the query counts where its dispatch changes form and
its blocks end, for every output count's path and several grid shapes, against
the oracle (1e-10 relative, the stated tolerance of the FP64 interpolant: an
exact linear identity up to rounding)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from oracle import grid as ogrid  # noqa: E402
from oracle import interp as ointerp  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(d, L, k, Q, seed):
    lo, hi = synth.box(d)
    og = ogrid.Grid(d, L, lo, hi)
    f = np.random.default_rng(seed).standard_normal((og.M, k))
    xq = synth.mixed_queries(Q, lo, hi, seed=seed + 1)
    n = min(Q, og.M, 20)
    xq[:n] = og.x[:n]                      # exact nodes among the queries
    if Q > 40:
        xq[n:n + 8] *= 1.2                 # outside the box
    return sg.Grid(d, L, lo, hi), og, f, xq


@pytest.mark.parametrize("Q", [1, 4, 31, 33, 608, 609, 2432, 2433, 3242, 3243, 6485, 10000])
def test_counts_where_the_form_changes(Q):
    g, og, f, xq = _case(6, 2, 3, Q, 100)
    S = sg.Surplus(g, torch.as_tensor(f, device="cuda"))
    u = sg.eval_feedback(S, torch.as_tensor(xq, device="cuda")).cpu().numpy()
    ref = ointerp.eval_surplus(og, ointerp.surpluses(og, f), xq)
    assert np.max(np.abs(u - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("d,L,k", [(1, 7, 1), (2, 6, 2), (3, 5, 4), (4, 4, 6), (5, 3, 7), (8, 2, 3), (7, 1, 16),
                                   (6, 0, 2), (2, 8, 5)])
@pytest.mark.parametrize("Q", [37, 5001])
def test_shapes(d, L, k, Q):
    g, og, f, xq = _case(d, L, k, Q, 7 * d + L)
    if Q > 40 and L > 4:
        xq = np.clip(xq, *synth.box(d))    # high degrees outside the box are ill-conditioned
    S = sg.Surplus(g, torch.as_tensor(f, device="cuda"))
    xd = torch.as_tensor(xq, device="cuda")
    if 8 * d * ((1 << L) + 1) * 128 > 200 * 1024:
        with pytest.raises(sg.SGError, match="level too high"):
            sg.eval_feedback(S, xd)
        return
    u = sg.eval_feedback(S, xd).cpu().numpy()
    ref = ointerp.eval_surplus(og, ointerp.surpluses(og, f), xq)
    assert np.max(np.abs(u - ref)) <= 1e-10 * np.max(np.abs(ref))
