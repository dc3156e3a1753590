"""Bodies of every make are accepted, alone (one block per body shape) and in
pairs (one block over all blobs), and their solves converge: filled cubes, a
plate, a rod, a ball, a filled shell, overlapping shells, with both kernels.
The true residual is formed with the saddle operator."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from test_pair_definite import ball, lattice  # noqa: E402

pytestmark = pytest.mark.gpu

S42 = workloads.icosahedral_shell(42, 2.5)
SHAPES = {
    "cube4": lattice((4, 4, 4), 1.5),
    "cube5": lattice((5, 5, 5), 1.0),
    "plate": lattice((1, 14, 14), 1.0),
    "rod": lattice((2, 2, 10), 1.0),
    "ball": ball(3.0, 1.1),
    "filled": np.concatenate([S42, workloads.icosahedral_shell(12, 1.2), [[0.0, 0, 0]]]),
    "overlap": np.concatenate([S42, S42[:, [1, 2, 0]] + [1.0, 0.3, 0.0]]),
}


@pytest.mark.parametrize("kernel", [3, 6])
@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("bodies", [1, 2])
def test_bodies_are_accepted_and_solved(name, bodies, kernel):
    import paper_1901_06427_gb300.binding as B
    rng = np.random.default_rng(17)
    ref = SHAPES[name] - SHAPES[name].mean(axis=0)
    gap = 2.0 * np.linalg.norm(ref, axis=1).max() + 2.0
    w = workloads.Workload(name="s", n=(int(gap * bodies) + 8, int(gap) + 8, int(gap) + 8), kernel=kernel)
    quat = workloads.configs.random_unit_quaternions(rng, bodies)
    at = [[4 + gap * (i + 0.5), 4 + gap / 2, 4 + gap / 2] for i in range(bodies)]
    w.bodies = [workloads.Body(ref, np.array(at[i]), quat[i]) for i in range(bodies)]
    g = B.grid_for(w, rtol=1e-8)
    assert g.body_block_info()[0] == (bodies == 2)
    FT = torch.tensor(rng.standard_normal(6 * bodies), device="cuda")
    U, info, x = g.mobility_solve(FT, return_x=True)
    b = torch.zeros(g.n_total, dtype=torch.float64, device="cuda")
    b[-6 * bodies:] = FT
    assert torch.isfinite(x).all()
    assert (torch.linalg.norm(b - g.apply_saddle(x)) / torch.linalg.norm(b)).item() < 1.01e-8
    assert torch.equal(U, x[-6 * bodies:])
