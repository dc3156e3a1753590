"""The exact level solve on axes of more than 48 points (folded line
transforms): with it both inner solves of the projection preconditioner are
exact, so its fluid block equals the projection method in FP32.  Odd and even
lines, every basis kind (walls, free-slip on one side or both, periodic),
both forms of the z pass, and lines that end just past a tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import operators, solve  # noqa: E402
import workloads  # noqa: E402
from gpu_common import rel  # noqa: E402

pytestmark = pytest.mark.gpu

F, T = False, True
CASES = {
    "x53": dict(n=(53, 9, 7)),
    "x64_periodic": dict(n=(64, 11, 6), periodic=(T, F, F)),
    "x49_periodic_odd": dict(n=(49, 7, 8), periodic=(T, F, F)),
    "x130_y_free": dict(n=(130, 9, 6), free_slip=(F, F, T, F, F, F)),
    "y65_mixed": dict(n=(10, 65, 6), free_slip=(F, F, T, F, F, T)),
    "z60_fwd_bwd": dict(n=(9, 8, 60), periodic=(T, F, F)),
    "z51_free_top": dict(n=(8, 9, 51), free_slip=(F, F, F, F, F, T)),
    "y66_periodic_xfree": dict(n=(7, 66, 8), periodic=(F, T, F), free_slip=(T, T, F, F, F, F)),
    "xy_long": dict(n=(70, 52, 5)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fluid_block_is_the_projection_method(name):
    from scipy.sparse.linalg import cg
    import paper_1901_06427_gb300.binding as B
    c = CASES[name]
    w = workloads.Workload(name=name, n=c["n"], periodic=c.get("periodic", (F, F, F)),
                           free_slip=c.get("free_slip", (F,) * 6))
    og = oracle.Grid(w.n, periodic=w.periodic, free_slip=w.free_slip)
    g = B.grid_for(w)
    lay = g.layout()
    nf, nc = lay[3], lay[4] - lay[3]
    r = np.random.default_rng(11).standard_normal(g.n_total)
    z = g.apply_preconditioner(torch.tensor(r, device="cuda")).cpu().numpy()
    vt = solve.viscous_solve(og, w.eta, r[None, :nf])[0]
    D, G = operators.divergence(og), operators.gradient(og)
    q = r[nf:nf + nc] + D @ vt
    phi, info = cg(-(D @ G), q - q.mean(), rtol=1e-13, maxiter=20000)
    assert info == 0
    # FP32 transforms: the gate of the short-line solve's test
    assert rel(z[:nf], vt + G @ phi) < 1e-4
    assert rel(z[nf:nf + nc], -w.eta * q) < 1e-4
