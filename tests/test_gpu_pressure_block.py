"""The pressure block as the solves apply it (rbfib_apply_preconditioner leaves
its drag term out), through a solve that stops after one iteration."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import operators, solve  # noqa: E402
from gpu_common import rel  # noqa: E402
from test_gpu_large_forms import B, ETA, neumann_solve  # noqa: E402, F401

pytestmark = pytest.mark.gpu
F, T = False, True


@pytest.mark.parametrize("free_slip,drag", [((F,) * 6, 12.0), ((F, T, F, T, F, T), 3.0)])
def test_pressure_block_of_the_solves(B, free_slip, drag):
    """One Krylov iteration returns a multiple of the preconditioned right-hand
    side, whose pressure in a solve is -eta (q + kappa phi): in a cube of side
    H, kappa is twice the drag 12 / H^2 between two no-slip walls, 3 / H^2 with
    one of them free-slip."""
    n = (14, 14, 14)
    og = oracle.Grid(n, free_slip=free_slip)
    g = B.Grid(n, eta=ETA, free_slip=free_slip, max_iter=1, rtol=1e-12)
    lay = g.layout()
    f = np.random.default_rng(5).standard_normal(lay[3])
    fd = torch.tensor(f, device="cuda")
    v = torch.empty(lay[3], dtype=torch.float64, device="cuda")
    pi = torch.empty(lay[4] - lay[3], dtype=torch.float64, device="cuda")
    info = B.SolveInfo()
    st = B.lib().rbfib_stokes_solve(g._h, *(ctypes.c_void_p(t.data_ptr()) for t in (fd, v, pi)), ctypes.byref(info))
    assert st == B.ENOCONV and info.iterations == 1
    vt = solve.viscous_solve(og, ETA, f[None])[0]
    D, G = operators.divergence(og), operators.gradient(og)
    q = D @ vt
    phi = neumann_solve(n, q)
    zv, zp = vt + G @ phi, -ETA * (q + 2.0 * drag / 14.0 ** 2 * phi)
    v, pi = v.cpu().numpy(), pi.cpu().numpy()
    scale = (v @ zv) / (zv @ zv)
    # FP32 transforms: the gate of the level solve's tests
    assert rel(v, scale * zv) < 1e-4
    assert rel(pi, scale * (zp - zp.mean())) < 1e-4
