"""The body block forms U = N (r_U + K^T M^-1 s) in FP64: with r_U the FP32
rounding of -K^T M^-1 s, U is N times that rounding, 2^-24 of the terms summed,
which FP32 sums or an FP32 matrix would bury.  One body in its own frame, no
fluid residual (J v = 0), so that the input of the block is r itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from test_gpu_body_solve import mobility  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blobs", [4, 12, 42, 162])
def test_rows_of_U_are_summed_in_fp64(blobs):
    import paper_1901_06427_gb300.binding as B
    if blobs == 4:
        ref = np.array([[1.0, 0, 0], [0, 1.1, 0], [0, 0, 0.9], [-0.6, -0.5, -0.4]])
    else:
        ref = workloads.icosahedral_shell(blobs, {12: 1.0, 42: 2.5, 162: 5.0}[blobs])
    w = workloads.Workload(name="b", n=(16, 16, 16))
    w.bodies = [workloads.Body(ref, np.array([8.1, 7.9, 8.0]), np.array([1.0, 0, 0, 0]))]
    g = B.grid_for(w)
    lay = g.layout()
    K = np.zeros((3 * blobs, 6))
    for i, d in enumerate(ref):
        K[3 * i:3 * i + 3, :3] = np.eye(3)
        K[3 * i:3 * i + 3, 3:] = [[0, d[2], -d[1]], [-d[2], 0, d[0]], [d[1], -d[0], 0]]
    P = np.linalg.solve(mobility(ref, 3, 1.0), K)
    N = np.linalg.inv(K.T @ P)
    x = np.zeros(g.n_total)
    s = np.random.default_rng(blobs).standard_normal(3 * blobs).astype(np.float32).astype(float)
    rU = (-P.T @ s).astype(np.float32).astype(float)
    x[lay[4]:lay[5]], x[lay[5]:] = s, rU
    U = g.apply_preconditioner(torch.tensor(x, device="cuda")).cpu().numpy()[lay[5]:]
    want = N @ (rU + P.T @ s)
    # the reference's own P is good to eps cond(M), 1e-12 of terms whose
    # rounding is 6e-8
    assert np.linalg.norm(U - want) < 1e-2 * np.linalg.norm(want)
