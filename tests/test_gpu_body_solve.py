"""The preconditioner's body block against a dense solve of its Schur
complement [-M K; K^T 0] (lambda, U) = -(r_lambda + J v), r_U with the pair
mobility of the source's tables: block sizes below, at and past the tiles of
the blocked inversion, coupled and per-body forms, both kernels."""
import numpy as np
import pytest
from scipy.interpolate import CubicSpline

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import ib, saddle  # noqa: E402
import workloads  # noqa: E402
from gpu_common import rel  # noqa: E402
from test_pair_mobility import tables  # noqa: E402

pytestmark = pytest.mark.gpu


def mobility(r, kw, eta):
    f, g = tables()[kw]
    a, shift = (1.47, 3e-5) if kw == 6 else (0.91, 2e-4)
    x = 0.25 * np.arange(25)
    tail = (lambda s: (1 + 2 * a * a / (3 * s * s)) / (8 * np.pi * s), lambda s: (1 - 2 * a * a / (3 * s * s)) / (4 * np.pi * s))
    d = r[:, None] - r[None]
    s = np.linalg.norm(d, axis=2)
    v = []
    for y, t in zip((f, g), tail):
        slope = (t(6 + 1e-5) - t(6 - 1e-5)) / 2e-5
        near = CubicSpline(x, y, bc_type=((1, 0.0), (1, slope)))(np.minimum(s, 6.0))
        v.append(np.where(s < 6.0, near, t(np.maximum(s, 1.0))))
    n = d / np.where(s > 0, s, 1.0)[..., None]
    M = v[0][..., None, None] * np.eye(3) + (v[1] - v[0])[..., None, None] * n[..., :, None] * n[..., None, :]
    return (M.transpose(0, 2, 1, 3).reshape(3 * len(r), -1) + shift * np.eye(3 * len(r))) / eta


@pytest.mark.parametrize("bodies,blobs,kernel,coupled", [
    (1, 12, 3, False), (1, 42, 6, False), (2, 12, 3, True), (8, 4, 3, True), (3, 12, 6, True), (11, 42, 3, True),
    (14, 12, 6, True), (43, 12, 3, False)])
def test_body_block(bodies, blobs, kernel, coupled):
    import paper_1901_06427_gb300.binding as B
    rng = np.random.default_rng(5)
    if blobs == 4:   # 3 N_bl = 96 = three whole tiles
        ref = np.array([[1.0, 0, 0], [0, 1.1, 0], [0, 0, 0.9], [-0.6, -0.5, -0.4]])
    else:
        ref = workloads.icosahedral_shell(blobs, 2.5 if blobs == 42 else 1.0)
    gap = 7.0 if blobs == 42 else 4.5
    side = int(np.ceil(bodies ** (1 / 3) - 1e-9))
    sites = np.array([(i, j, k) for i in range(side) for j in range(side) for k in range(side)][:bodies])
    n = (int(gap * (side - 1)) + 10,) * 3
    w = workloads.Workload(name="b", n=n, kernel=kernel, eta=1.3)
    quat = workloads.configs.random_unit_quaternions(rng, bodies)
    w.bodies = [workloads.Body(ref, 5.0 + gap * at + rng.uniform(-0.2, 0.2, 3), quat[i]) for i, at in enumerate(sites)]
    g = B.grid_for(w)
    assert g.body_block_info()[0] == coupled
    og = oracle.Grid(w.n, kernel=kernel)
    ob = saddle.Bodies(w.ref_blobs, w.blob_offsets, w.q, w.quat)
    lay = g.layout()
    x = rng.standard_normal(g.n_total)
    z = g.apply_preconditioner(torch.tensor(x, device="cuda")).cpu().numpy()
    r = ob.positions()
    s = x[lay[4]:lay[5]] + ib.interpolate(og, r, z[:lay[3]])
    K = np.zeros((3 * w.n_blobs, 6 * bodies))
    for p in range(bodies):
        for i in range(w.blob_offsets[p], w.blob_offsets[p + 1]):
            d = r[i] - w.q[p]
            K[3 * i:3 * i + 3, 6 * p:6 * p + 3] = np.eye(3)
            K[3 * i:3 * i + 3, 6 * p + 3:6 * p + 6] = [[0, d[2], -d[1]], [-d[2], 0, d[0]], [d[1], -d[0], 0]]
    M = mobility(r, kernel, w.eta)
    if not coupled:
        body = np.repeat(np.arange(bodies), 3 * blobs)
        M = np.where(body[:, None] == body[None], M, 0.0)
    X = np.linalg.inv(M)
    U = np.linalg.solve(K.T @ X @ K, x[lay[5]:] + K.T @ (X @ s))
    lam = X @ (K @ U - s)
    # FP32 inverse of M (condition up to about 2e4): eps x condition
    tol = 6e-8 * np.linalg.cond(M) * 4 + 1e-4
    assert rel(z[lay[4]:lay[5]], lam) < tol
    assert rel(z[lay[5]:], U) < tol
