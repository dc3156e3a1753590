"""Forms of the kernels that only larger grids select.
- The pipelined Stokes operator with 32 planes a block (four blocks per SM),
  every periodic axis, ragged last tiles in x, y and z, FP64 and FP32, against
  a plain torch operator, itself checked against the oracle on a small grid.
- The wide tile of the long-line passes (two blocks per SM), lines along every
  axis, both directions: velocity against the oracle's transforms, pressure
  against a cosine transform.
Gates as for the same operators on smaller grids."""
import numpy as np
import pytest
import scipy.fft as sfft

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import operators, saddle, solve  # noqa: E402
import workloads  # noqa: E402
from gpu_common import assert_close, rel, F32_MATVEC, F64_MATVEC  # noqa: E402

pytestmark = pytest.mark.gpu
F, T = False, True
ETA = 1.3


@pytest.fixture(scope="module")
def B():
    import paper_1901_06427_gb300.binding as binding
    binding.lib()
    return binding


def stokes(n, per, x):
    """(-eta LL v + G pi, -D v) on a MAC grid of spacing 1 with no-slip walls;
    arrays are (z, y, x), the walls' own faces are left out."""
    cells = (n[2], n[1], n[0])
    shape = [tuple(n[ax] - (ax == a and not per[ax]) for ax in (2, 1, 0)) for a in range(3)]
    parts = torch.split(x, [int(np.prod(s)) for s in shape] + [int(np.prod(cells))])
    v, p = [q.reshape(s) for q, s in zip(parts, shape)], parts[3].reshape(cells)

    def shifts(f, dim, wall):   # neighbours below and above; wall: ghost as a multiple of the end
        if wall is None:
            return torch.roll(f, 1, dim), torch.roll(f, -1, dim)
        m = f.shape[dim]
        first, last = f.narrow(dim, 0, 1), f.narrow(dim, m - 1, 1)
        return (torch.cat([wall * first, f.narrow(dim, 0, m - 1)], dim),
                torch.cat([f.narrow(dim, 1, m - 1), wall * last], dim))

    out, div = [], torch.zeros_like(p)
    for a in range(3):
        lap = -6.0 * v[a]
        for ax in range(3):
            lo, hi = shifts(v[a], 2 - ax, None if per[ax] else (0.0 if ax == a else -1.0))
            lap = lap + lo + hi
        dim = 2 - a
        if per[a]:
            out.append(-ETA * lap + p - torch.roll(p, 1, dim))
            div = div + torch.roll(v[a], -1, dim) - v[a]
        else:
            out.append(-ETA * lap + p.narrow(dim, 1, n[a] - 1) - p.narrow(dim, 0, n[a] - 1))
            zero = torch.zeros_like(p.narrow(dim, 0, 1))
            faces = torch.cat([zero, v[a], zero], dim)
            div = div + faces.narrow(dim, 1, n[a]) - faces.narrow(dim, 0, n[a])
    return torch.cat([o.reshape(-1) for o in out] + [-div.reshape(-1)])


def neumann_solve(n, q):
    """phi of mean zero with -D G phi = q between walls, by cosine transforms."""
    lam = [2.0 - 2.0 * np.cos(np.pi * np.arange(m) / m) for m in n]
    den = lam[2][:, None, None] + lam[1][None, :, None] + lam[0]
    den[0, 0, 0] = 1.0
    c = sfft.dctn(q.reshape(n[::-1]), type=2) / den
    c[0, 0, 0] = 0.0
    return sfft.idctn(c, type=2).ravel()


def empty(n, per, free_slip=(F,) * 6):
    return workloads.Workload(name="empty", n=n, periodic=per, free_slip=free_slip, eta=ETA)


@pytest.mark.parametrize("per", [(F, F, F), (T, F, F), (F, T, F), (F, F, T), (T, T, F), (F, T, T), (T, F, T)])
def test_stokes_operator_with_32_planes_a_block(B, per):
    gen = torch.Generator("cuda").manual_seed(3)
    small = (7, 6, 5)
    og = oracle.Grid(small, periodic=per)
    none = saddle.Bodies(np.zeros((0, 3)), [0], np.zeros((0, 3)), np.zeros((0, 4)))
    xs = np.random.default_rng(1).standard_normal(og.N_f + og.N_c)
    assert rel(stokes(small, per, torch.tensor(xs)).numpy(), saddle.apply(og, none, ETA, xs)) < 1e-14
    n = (65, 33, 1290)   # 3 x 5 tiles of 32 x 8, 41 chunks of 32 planes
    g = B.grid_for(empty(n, per))
    x = torch.randn(g.n_total, dtype=torch.float64, device="cuda", generator=gen)
    lay = g.layout()
    for dtype, gate in ((torch.float64, F64_MATVEC), (torch.float32, F32_MATVEC)):
        xt = x.to(dtype)
        y, y0 = g.apply_saddle(xt).double().cpu().numpy(), stokes(n, per, xt.double()).cpu().numpy()
        for lo, hi in zip(lay[:4], lay[1:5]):
            assert_close(y[lo:hi], y0[lo:hi], gate, str(dtype))


@pytest.mark.parametrize("n,per,free_slip", [((130, 90, 52), (F, F, F), (F,) * 6),
                                             ((129, 91, 51), (T, F, F), (F,) * 6),
                                             ((131, 90, 53), (F, T, F), (F, T, F, F, T, F)),
                                             ((150, 100, 46), (F, F, F), (F, F, T, T, F, F))])
def test_wide_line_tiles_velocity(B, n, per, free_slip):
    w = empty(n, per, free_slip)
    og = oracle.Grid(n, periodic=per, free_slip=free_slip)
    g = B.grid_for(w)
    lay = g.layout()
    r = np.random.default_rng(11).standard_normal(g.n_total)
    vt = solve.viscous_solve(og, w.eta, r[None, :lay[3]])[0]
    # with r_pi = -D v~ the potential vanishes and the block returns v~
    r[lay[3]:] = -(operators.divergence(og) @ vt)
    z = g.apply_preconditioner(torch.tensor(r, device="cuda")).cpu().numpy()
    for lo, hi in zip(lay[:3], lay[1:4]):
        assert rel(z[lo:hi], vt[lo:hi]) < 1e-4


def test_wide_line_tiles_pressure(B):
    n = (130, 130, 131)
    w = empty(n, (F, F, F))
    og = oracle.Grid(n)
    g = B.grid_for(w)
    lay = g.layout()
    r = np.zeros(g.n_total)
    q = np.random.default_rng(12).standard_normal(n[::-1])
    r[lay[3]:] = (q - q.mean()).ravel()
    phi = neumann_solve(n, r[lay[3]:])
    z = g.apply_preconditioner(torch.tensor(r, device="cuda")).cpu().numpy()
    assert rel(z[:lay[3]], operators.gradient(og) @ phi) < 1e-4
    assert rel(z[lay[3]:], -w.eta * r[lay[3]:]) < 1e-4
