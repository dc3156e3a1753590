"""A grid whose set_bodies call failed can be used: bodies that are refused
leave it as it was, and where the failure comes while the configuration is
being built (two blobs of the coupled block at one place) it is left without
bodies, every size with its buffers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads  # noqa: E402

pytestmark = pytest.mark.gpu

TRIANGLE = np.array([[0.0, 0, 0], [1.2, 0, 0], [0, 1.1, 0]])


@pytest.fixture(scope="module")
def B():
    import paper_1901_06427_gb300.binding as binding
    binding.lib()
    return binding


def spheres(bodies):
    shell = workloads.icosahedral_shell(42, 2.5)
    return (42 * np.arange(bodies + 1), np.tile(shell, (bodies, 1)),
            np.array([[5.0 + 7 * i, 5.0, 5.0] for i in range(bodies)]), np.tile([1.0, 0, 0, 0], (bodies, 1)))


@pytest.mark.parametrize("precision", ["FP64", "FP32_REFINED"])
def test_refused_bodies_leave_the_grid_as_it_was(B, precision):
    g = B.Grid((10, 10, 10), precision=getattr(B, precision), rtol=1e-9)
    g.set_bodies([0, 3], TRIANGLE, [[5.0, 5.0, 5.0]], [[1.0, 0, 0, 0]])
    lay = g.layout()
    FT = torch.tensor([1.0, -2.0, 0.5, 0.3, 0.2, -0.7], dtype=torch.float64, device="cuda")
    U0, i0 = g.mobility_solve(FT)
    big = np.concatenate([workloads.icosahedral_shell(162, 3.0), [[1.0, 1, 1], [1.0, 1, 1]]])   # two blobs at one place
    with pytest.raises(B.RbfibError) as e:
        g.set_bodies([0, 164], big, [[5.0, 5.0, 5.0]], [[1.0, 0, 0, 0]])
    assert e.value.code == B.EINVAL
    assert g.layout() == lay and (g.n_bodies, g.n_blobs) == (1, 3)
    U1, i1 = g.mobility_solve(FT)
    # the same solve again: atomic sums in another order, the solver's tolerance
    assert torch.linalg.norm(U1 - U0).item() < 1e-6 * torch.linalg.norm(U0).item()
    assert abs(i1["iterations"] - i0["iterations"]) <= 1


def test_failure_in_the_coupled_block_leaves_no_bodies(B):
    g = B.Grid((24, 10, 10), rtol=1e-9)
    g.set_bodies([0, 3], TRIANGLE, [[5.0, 5.0, 5.0]], [[1.0, 0, 0, 0]])
    off, ref, q, quat = spheres(2)
    with pytest.raises(B.RbfibError) as e:
        g.set_bodies(off, ref, q[[0, 0]], quat)   # one sphere on top of the other
    assert e.value.code == B.EINTERNAL
    lay = g.layout()
    assert lay[4] == lay[5] == lay[6] and (g.n_bodies, g.n_blobs) == (0, 0)
    f = torch.randn(lay[3], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    v0, _, _ = g.stokes_solve(f)
    z = g.apply_preconditioner(torch.ones(lay[6], dtype=torch.float64, device="cuda"))
    fresh = B.Grid((24, 10, 10), rtol=1e-9)
    v1, _, _ = fresh.stokes_solve(f)
    assert torch.isfinite(z).all()
    assert torch.linalg.norm(v0 - v1).item() < 1e-6 * torch.linalg.norm(v1).item()
    g.set_bodies(*spheres(2))
    U, info = g.mobility_solve(torch.ones(12, dtype=torch.float64, device="cuda"))
    assert torch.isfinite(U).all() and info["rel_residual"] < 1e-9
