"""Which way the coupled block of two 42-blob spheres (252 rows, the largest
that may start warm) is inverted after a step: small moves take Newton-Schulz
steps from the rotated inverse, moves of a Brownian time step the blocked
inversion.  Either way the block is that of a fresh grid at the same place."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,warm", [(1e-6, True), (0.05, False)])
def test_choice_after_a_step(dt, warm):
    import paper_1901_06427_gb300.binding as B
    w = workloads.two_sphere_cavity(steps=1)
    g = B.grid_for(w)
    q, quat = (torch.tensor(np.asarray(v, dtype=np.float64).ravel(), device="cuda") for v in (w.q, w.quat))
    p = B.sem_params(w.potentials, dt=dt, kT=1.0)
    assert g.sem_step(p, w.seed, 0, 0, q, quat)[0] == 0   # rebuilt where it was: always warm
    n0 = g.body_block_info()[1]
    q1, quat1 = q.clone(), quat.clone()
    assert g.sem_step(p, w.seed, 1, 0, q, quat)[0] == 0   # rebuilt at (q1, quat1)
    assert g.body_block_info()[1] == n0 + warm
    fresh = B.Grid(w.n, h=w.h, eta=w.eta, periodic=w.periodic, wall_vel=w.wall_vel)
    fresh.set_bodies(w.blob_offsets, w.ref_blobs, q1.reshape(-1, 3).cpu().numpy(), quat1.reshape(-1, 4).cpu().numpy())
    r = torch.randn(g.n_total, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    za, zb = g.apply_preconditioner(r), fresh.apply_preconditioner(r)
    # FP32 inverses of a matrix of condition up to 1e4
    assert (torch.linalg.norm(za - zb) / torch.linalg.norm(zb)).item() < 2e-3
