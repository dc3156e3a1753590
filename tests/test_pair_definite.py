"""The blob mobility of the body block (csrc/pair_mobility.cuh) is positive
definite for any distinct blobs, as the grid's own mobility is: bodies whose
blobs fill a volume or a plane, overlapping bodies, dense clusters and packed
suspensions, with the smallest raise of the diagonal."""
import numpy as np
import pytest

import workloads
from test_gpu_body_solve import mobility


def lattice(n, h):
    return h * np.stack(np.meshgrid(*[np.arange(k) for k in n], indexing="ij"), axis=-1).reshape(-1, 3).astype(float)


def ball(radius, h):
    m = int(radius / h)
    p = lattice((2 * m + 1,) * 3, h) - m * h
    return p[np.linalg.norm(p, axis=1) <= radius + 1e-9]


def packed(bodies, blobs, radius, pitch):
    """Shells of random orientation on a cubic lattice, a little off it."""
    from scipy.spatial.transform import Rotation
    rng = np.random.default_rng(5)
    ref = workloads.icosahedral_shell(blobs, radius)
    side = int(np.ceil(bodies ** (1 / 3) - 1e-9))
    at = pitch * lattice((side,) * 3, 1.0)[:bodies] + rng.uniform(-0.2, 0.2, (bodies, 3))
    return np.concatenate([a + ref @ Rotation.random(random_state=rng).as_matrix().T for a in at])


def shapes():
    rng = np.random.default_rng(1)
    s42 = workloads.icosahedral_shell(42, 2.5)
    out = {"overlap": np.concatenate([s42, s42[:, [1, 2, 0]] + [1.0, 0.3, 0.0]]),
           "filled shell": np.concatenate([s42, workloads.icosahedral_shell(12, 1.2), [[0.0, 0, 0]]]),
           "cluster": rng.uniform(-1.0, 1.0, (120, 3)), "cloud": rng.uniform(-3.0, 3.0, (300, 3)),
           "twins": np.concatenate([s42, s42 + 1e-6])}
    for n, h in ((4, 1.25), (4, 1.5), (5, 0.9), (5, 1.5), (6, 1.0), (7, 1.1), (8, 0.9)):
        out[f"cube {n} at {h}"] = lattice((n,) * 3, h)
    for n, h in ((12, 1.1), (14, 0.75), (16, 1.0), (16, 1.25)):
        out[f"plate {n} at {h}"] = lattice((1, n, n), h)
    for h in (0.75, 1.0, 1.25):
        out[f"slab at {h}"], out[f"rod at {h}"] = lattice((2, 8, 8), h), lattice((2, 2, 10), h)
        out[f"ball at {h}"] = ball(3.0, h)
    for bodies, blobs, radius, pitch in ((3, 12, 1.0, 4.5), (14, 12, 1.0, 4.5), (24, 12, 1.0, 4.5), (11, 42, 2.5, 7.0)):
        out[f"{bodies} shells of {blobs}"] = packed(bodies, blobs, radius, pitch)
    return out


SHAPES = shapes()


@pytest.mark.parametrize("kernel", [3, 6])
@pytest.mark.parametrize("name", list(SHAPES))
def test_smallest_eigenvalue_is_positive(name, kernel):
    assert np.linalg.eigvalsh(mobility(SHAPES[name], kernel, 1.0))[0] > 0.0
