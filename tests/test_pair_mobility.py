"""The pair functions of the body block (csrc/pair_mobility.cuh) against a
spectral Stokes solution on the staggered grid, with the oracle's kernels."""
import os
import re

import numpy as np
import pytest

from oracle.kernel import kernel

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_06427_gb300", "csrc",
                   "pair_mobility.cuh")


def tables():
    """{3: (f, g), 6: (f, g)} at r = 0, 1/4, ..., 6 as the source has them."""
    body = open(SRC).read()
    out = {}
    for kw, name in ((3, "three"), (6, "six")):
        text = re.search(r"static const double %s\[2\]\[kPairKnots\] = \{(.*?)\};" % name, body, re.S).group(1)
        out[kw] = np.array([float(v) for v in re.findall(r"\d+\.\d+", text)]).reshape(2, 25)
    return out


@pytest.mark.parametrize("kw", [3, 6])
def test_pair_functions_are_the_grids_response(kw):
    """A unit force spread at a few offsets in a periodic box of 40 cells; the
    images shift every velocity by 2.837 / (6 pi L), and by O(r^2 / L^3)."""
    n, offsets = 40, 4
    phi, _, k, first = kernel(kw)
    rng = np.random.default_rng(3)
    th = 2 * np.pi * np.fft.fftfreq(n)
    K = [2 * np.sin(th / 2).reshape([-1 if a == b else 1 for b in range(3)]) for a in range(3)]
    P = [np.exp(1j * th / 2).reshape([-1 if a == b else 1 for b in range(3)]) for a in range(3)]
    k2 = K[0] ** 2 + K[1] ** 2 + K[2] ** 2
    k2[0, 0, 0] = np.inf

    def weights(x, a):
        at, w = [], []
        for ax in range(3):
            s = x[ax] - (0.0 if ax == a else 0.5)
            p = first(np.array([s]))[0] + np.arange(k)
            at.append(p % n)
            w.append(phi(s - p))
        return np.ix_(*at), np.einsum("i,j,k->ijk", *w)

    rs = [0.0, 0.5, 1.0, 2.0, 3.5]
    got = np.zeros((2, len(rs)))
    for _ in range(offsets):
        x0 = n / 2 + rng.uniform(0, 1, 3)
        v = [[None] * 3 for _ in range(3)]
        for b in range(3):
            f = np.zeros((n, n, n))
            at, w = weights(x0, b)
            f[at] = w
            fh = np.fft.fftn(f) * P[b]
            for a in range(3):
                u = ((fh if a == b else 0) - K[a] * K[b] * fh / k2) / k2
                v[a][b] = np.fft.ifftn(u * np.conj(P[a])).real
        for _ in range(8):
            d = rng.standard_normal(3)
            d /= np.linalg.norm(d)
            for j, r in enumerate(rs):
                G = np.zeros((3, 3))
                for a in range(3):
                    at, w = weights(x0 + r * d, a)
                    for b in range(3):
                        G[a, b] = np.sum(v[a][b][at] * w)
                along = d @ G @ d
                got[:, j] += np.array([(np.trace(G) - along) / 2, along]) / (8 * offsets)
    got += 2.837297 / (6 * np.pi * n)
    want = tables()[kw][:, [int(4 * r) for r in rs]]
    # 32 draws: the three-point kernel varies by about 1% with the offset; the
    # images' next order is r^2 / L^3, below 2e-4 of 1 / 8
    assert np.max(np.abs(got - want) / want) < 0.012
