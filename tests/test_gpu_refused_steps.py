"""FP64 solves whose full Newton step is refused, or whose tree direction has lost
digits: the elimination with full partial pivoting forms the direction of such
a node, its full step is tried, in every launch form and with damping on or
off, and it costs what it should."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from oracle import lobatto  # noqa: E402
from oracle import problems as oprob  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu
LO, HI = synth.box(6)
A4 = lobatto.tableau()[0]


def cuda(x, dtype=torch.float64):
    return torch.as_tensor(np.asarray(x), dtype=dtype, device="cuda")


def _indefinite_lq():
    params = synth.lq_params(0)
    params.A = np.diag([3.0, -1.0, -1.2, -0.8, -0.5, -0.3]) + 0.02 * params.A
    params.B = 0.3 * params.B
    params.Q = np.diag([-1.0, 1.0, 1.0, 1.0, 1.0, 1.0])
    return params


def _interval_det(pr, h):
    """det of the block that one interval's scattering form inverts."""
    J = oprob.rhs_jacobian(pr, np.zeros((12, 1)))[:, :, 0]
    blk = [[-h * A4[k, j] * J + (np.eye(12) if j == k else 0) - (np.eye(12) if j == 0 else 0) for j in range(4)]
           for k in (1, 2, 3)]
    inner = np.block([[blk[0][1], blk[0][2]], [blk[1][1], blk[1][2]]])
    outer = np.block([[blk[0][0], blk[0][3]], [blk[1][0], blk[1][3]]])
    st = np.hstack([blk[2][0], blk[2][3]]) - np.hstack([blk[2][1], blk[2][2]]) @ np.linalg.solve(inner, outer)
    return np.linalg.det(np.hstack([st[:, 12:18], st[:, 6:12]]))


def _singular_width(pr):
    hs = np.linspace(0.05, 4.0, 800)
    d = np.array([_interval_det(pr, h) for h in hs])
    k = np.flatnonzero(d[:-1] * d[1:] < 0)
    lo, hi = hs[k[0]], hs[k[0] + 1]
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if not lo < mid < hi:
            break
        lo, hi = (mid, hi) if _interval_det(pr, lo) * _interval_det(pr, mid) > 0 else (lo, mid)
    return lo


@pytest.mark.parametrize("damping", [True, False])
def test_full_step_where_the_tree_loses_digits(damping):
    """Mesh widths 2^-8 .. 2^-45 (relative) from the one at which no interval has a
    scattering form: the linear problem's one Newton step is taken at full
    length whatever the tree made of it (a second one polishes)."""
    params = _indefinite_lq()
    h = _singular_width(oprob.make(params)) * (1.0 + 2.0 ** -np.arange(8.0, 46.0, 0.5))
    n, N = h.size, 3
    X0 = synth.uniform_queries(n, LO, HI, seed=81)
    res = sg.solve_bvps(sg.problem_from(params), cuda(X0), cuda(N * h), N, tol=1e-8, damping=damping)
    assert torch.all(res["status"] == sg.CONVERGED)
    assert int(res["iters"].max()) <= 2, res["iters"].cpu().numpy()


def _far(n, scale, seed=17):
    return cuda(scale * np.random.default_rng(seed).uniform(LO, HI, (n, 6)))


@pytest.mark.parametrize("damping", [True, False])
def test_launch_forms_agree_where_steps_are_refused(damping):
    """States up to 1.5 times the box: some nodes take damped steps.  Host loop,
    one graph, a graph per mesh size and the pool give the same bits, and the
    persistent form (elimination throughout) the same roots."""
    n, N = 90, 128
    prob = sg.problem_from(synth.attitude_params(0))
    X = _far(n, 1.5)
    T = 20.0
    ref = sg.solve_bvps(prob, X, T, N, damping=damping, graph=0)
    assert int((ref["iters"] > 6).sum()) > 0          # some were refused
    for graph in (1, 2):
        got = sg.solve_bvps(prob, X, T, N, damping=damping, graph=graph)
        for key in ("lambda0", "u0", "V", "status", "iters"):
            assert torch.equal(got[key].nan_to_num(), ref[key].nan_to_num()), (graph, key)
    pool = sg.SolverPool(prob, n, N, precision=sg.PREC_FP64, damping=damping)
    slots = pool.admit(X, T, N)
    while pool.iterate():
        pass
    got = pool.collect(slots)
    for key in ("lambda0", "u0", "V", "status", "iters"):
        assert torch.equal(got[key].nan_to_num(), ref[key].nan_to_num()), ("pool", key)
    if damping:
        per = sg.solve_bvps(prob, X, T, N, persistent=True)
        assert torch.equal(per["status"], ref["status"]) and torch.all(ref["status"] == sg.CONVERGED)
        assert torch.max(torch.abs(per["lambda0"] - ref["lambda0"])) <= 1e-6 * torch.max(torch.abs(per["lambda0"]))


def _ms(fn):
    fn()
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def test_refused_steps_cost():
    """85 nodes, one graph: an iteration with refused steps (states of twice the box;
    a dozen nodes use up 50 iterations) takes at most four times as long as one
    without (it took seven and a half times when a block did a node's
    elimination on its own; the elimination itself and its halvings are worth two)."""
    n, N = 85, 128
    prob = sg.problem_from(synth.attitude_params(0))
    per = []
    for X in (_far(n, 1.0), _far(n, 2.0)):
        keep = dict(n_max=N, workspace=torch.empty(sg.workspace_bytes(n, N, sg.PREC_FP64), dtype=torch.uint8,
                                                   device="cuda"))
        out = sg.solve_bvps(prob, X, 20.0, N, graph=1, **keep)
        ms = _ms(lambda: sg.solve_bvps(prob, X, 20.0, N, graph=1, out=out, **keep))
        per.append(ms / int(out["iters"].max()))
    assert per[1] <= 4.0 * per[0], per
