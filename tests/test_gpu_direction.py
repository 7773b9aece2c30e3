"""The FP64 form's Newton direction (scattering tree over the intervals) at the
mesh sizes where its tiles end, and at a mesh whose single intervals have no
scattering form (the marked nodes' path).

On the linear-quadratic problem the discrete solution is lambda(0) = P0 x0 with
P0 from the discrete Riccati recursion.  Tolerance: one FP64 elimination of a
well-conditioned system (the stated 1e-10 relative of the other LQ tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import synth  # noqa: E402
from oracle import bvp as obvp  # noqa: E402
from oracle import lobatto  # noqa: E402
from oracle import problems as oprob  # noqa: E402
from oracle import riccati  # noqa: E402
from paper_1507_04769_gb300 import sg  # noqa: E402

pytestmark = pytest.mark.gpu

LO, HI = synth.box(6)
A4 = lobatto.tableau()[0]


def cuda(x, dtype=torch.float64):
    return torch.as_tensor(np.asarray(x), dtype=dtype, device="cuda")


@pytest.mark.parametrize("n", [1, 160, 700])      # the three block sizes of the tree
def test_lq_matches_riccati_at_tile_edges(n):
    params = synth.lq_params(0)
    pr = oprob.make(params)
    sizes = [1, 2, 3, 7, 8, 9, 15, 16, 17, 31, 33, 63, 65, 129]
    N = np.array([sizes[(k + 9) % len(sizes)] for k in range(n)])
    T = 10.0 * N / N.max()
    X0 = synth.uniform_queries(n, LO, HI, seed=77)
    res = sg.solve_bvps(sg.problem_from(params), cuda(X0), cuda(T), cuda(N, torch.int32), tol=1e-12)
    assert torch.all(res["status"] == sg.CONVERGED)
    lam = res["lambda0"].cpu().numpy()
    for size in sorted(set(N.tolist())):
        k = np.flatnonzero(N == size)
        ref = X0[k] @ riccati.riccati_p0(pr, float(T[k[0]]), int(size), discrete=True).T
        assert np.max(np.abs(lam[k] - ref)) <= 1e-10 * np.max(np.abs(ref)), size


def _interval_det(pr, h):
    """det of the block that one interval's scattering form inverts."""
    J = oprob.rhs_jacobian(pr, np.zeros((12, 1)))[:, :, 0]
    blk = [[-h * A4[k, j] * J + (np.eye(12) if j == k else 0) - (np.eye(12) if j == 0 else 0) for j in range(4)]
           for k in (1, 2, 3)]
    inner = np.block([[blk[0][1], blk[0][2]], [blk[1][1], blk[1][2]]])
    outer = np.block([[blk[0][0], blk[0][3]], [blk[1][0], blk[1][3]]])
    st = np.hstack([blk[2][0], blk[2][3]]) - np.hstack([blk[2][1], blk[2][2]]) @ np.linalg.solve(inner, outer)
    return np.linalg.det(np.hstack([st[:, 12:18], st[:, 6:12]]))


def test_interval_without_scattering_form():
    """A mesh width at which (x_{i+1}, lambda_i) does not follow from (x_i,
    lambda_{i+1}) on any single interval, while the boundary value problem is
    regular: those nodes take the elimination with full partial pivoting."""
    params = synth.lq_params(0)
    # one growing mode with a negative weight: the determinant changes sign
    params.A = np.diag([3.0, -1.0, -1.2, -0.8, -0.5, -0.3]) + 0.02 * params.A
    params.B = 0.3 * params.B
    params.Q = np.diag([-1.0, 1.0, 1.0, 1.0, 1.0, 1.0])
    pr = oprob.make(params)
    hs = np.linspace(0.05, 4.0, 800)
    d = np.array([_interval_det(pr, h) for h in hs])
    k = np.flatnonzero(d[:-1] * d[1:] < 0)
    assert k.size, "no singular width found"
    lo, hi = hs[k[0]], hs[k[0] + 1]
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if not lo < mid < hi:
            break
        lo, hi = (mid, hi) if _interval_det(pr, lo) * _interval_det(pr, mid) > 0 else (lo, mid)
    X0 = synth.uniform_queries(5, LO, HI, seed=78)
    N = 3
    res = sg.solve_bvps(sg.problem_from(params), cuda(X0), N * lo, N, tol=1e-9)
    assert torch.all(res["status"] == sg.CONVERGED)
    for j in range(5):
        s = obvp.solve(pr, X0[j], N * lo, N)
        assert np.max(np.abs(res["lambda0"][j].cpu().numpy() - s.lambda0)) <= 1e-8 * np.max(np.abs(s.lambda0))


def test_tree_leaves_by_blocks_give_the_same_bits():
    """Fewer than 304 nodes run the tree's lowest levels in blocks of their own:
    the same compositions, so the same results to the last bit as in a solve of
    more nodes."""
    params = synth.lq_params(1)
    n, more = 303, 305
    sizes = [1, 15, 16, 17, 32, 33, 47, 64, 100, 129]
    N = np.array([sizes[k % len(sizes)] for k in range(more)])
    T = 10.0 * N / N.max()
    X0 = synth.uniform_queries(more, LO, HI, seed=79)
    few = sg.solve_bvps(sg.problem_from(params), cuda(X0[:n]), cuda(T[:n]), cuda(N[:n], torch.int32))
    many = sg.solve_bvps(sg.problem_from(params), cuda(X0), cuda(T), cuda(N, torch.int32))
    for key in ("lambda0", "u0", "V", "status", "iters"):
        assert torch.equal(few[key], many[key][:n]), key


@pytest.mark.parametrize("make", [synth.attitude_params, synth.example1_params, synth.example2_params])
def test_attitude_zeros_against_general_elimination(make):
    """The attitude family's condensation leaves out the Jacobian's structural
    zeros; the persistent form eliminates the whole blocks.  Both converge
    quadratically to |F| <= 1e-12, so lambda(0) agrees far below 1e-8 of its
    size, and the statuses are the same."""
    params = make()
    sizes = [1, 2, 7, 8, 9, 24, 33]
    n = len(sizes)
    X0 = 0.3 * synth.uniform_queries(n, LO, HI, seed=80)
    N = np.array(sizes)
    T = np.minimum(0.15 * N, 4.0)
    prob = sg.problem_from(params)
    a = sg.solve_bvps(prob, cuda(X0), cuda(T), cuda(N, torch.int32), tol=1e-12)
    b = sg.solve_bvps(prob, cuda(X0), cuda(T), cuda(N, torch.int32), tol=1e-12, persistent=True)
    assert torch.equal(a["status"], b["status"])
    la, lb = a["lambda0"], b["lambda0"]
    assert torch.all(a["status"] == sg.CONVERGED)
    assert torch.max(torch.abs(la - lb)) <= 1e-8 * torch.max(torch.abs(lb))
