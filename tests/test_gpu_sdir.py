"""GPU: u.S x over tiles of low sites (shared memory) and high sites (other tiles),
against the definition applied site by site in FP64, for every way the sites
split: one tile, ragged tiles, spins up to 15/2, group remainders in R.

Tolerance: 2 n ladder terms and three products a value: 4 n units roundoff of
the sum of the terms' magnitudes (2^-24 or 2^-53)."""
import numpy as np
import pytest

import ftlm_workloads as W
import oracle
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev, osys, to_dev

pytestmark = pytest.mark.gpu


def plain(two_s, u, x):
    """(u.S x, sum of the terms' magnitudes), site by site"""
    y, mag = np.zeros_like(x), np.zeros(x.shape)
    a = 0.5 * (u[0] - 1j * u[1])
    stride = 1
    for t in two_s:
        s, q = t / 2, t + 1
        m = np.arange(q) - s
        v = x.reshape(-1, q, stride, x.shape[1])
        o = u[2] * m[None, :, None, None] * v
        g = np.abs(o)
        up = np.sqrt(s * (s + 1) - m[:-1] * (m[:-1] + 1))[None, :, None, None]
        o[:, 1:] += a * up * v[:, :-1]
        o[:, :-1] += np.conj(a) * up * v[:, 1:]
        g[:, 1:] += np.abs(a * up * v[:, :-1])
        g[:, :-1] += np.abs(a * up * v[:, 1:])
        y += o.reshape(x.shape)
        mag += g.reshape(x.shape)
        stride *= q
    return y, mag


@pytest.mark.parametrize("two_s", [[1], [2, 1], [15, 15, 3], [1] * 10, [1] * 13, [2] * 8, [5, 4, 4, 4, 4, 4], [3, 1, 2, 5, 1, 2, 4]])
@pytest.mark.parametrize("R", [1, 2, 3, 5, 8])
def test_sdir_matches_definition(two_s, R, rng):
    s = F.System(two_s, B=(0.3, 0.1, 0.5))
    u = np.array([0.4, -0.7, 0.59])
    u /= np.linalg.norm(u)
    x = rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R))
    for dtype, eps in (("c64", 2.0 ** -24), ("c128", 2.0 ** -53)):
        xd, yd = to_dev(x, dtype), empty_dev((s.dim, R), dtype)
        F.apply_sdir(s, xd, yd, R, dtype, u=u)
        ref, mag = plain(two_s, u, xd.cpu().numpy().astype(np.complex128))
        err = np.abs(yd.cpu().numpy() - ref)
        assert np.all(err <= (4 * len(two_s) + 8) * eps * mag)
    s.close()


@pytest.mark.parametrize("make", [lambda B: W.chain(5, Bdir=B), lambda B: W.square_lattice(13, 1, Bdir=B)])
@pytest.mark.parametrize("Bdir", [(0, 0, 1), (1, 0, 0), (0, 1, 0)])
def test_runs_along_the_axes(make, Bdir):
    """The projections p of a run whose u lies along z (no neighbours) or an axis of
    the plane; after four steps 1e-12 of the largest, the rounding of the steps' sums."""
    w = make(Bdir)
    s = F.System.from_dict(w)
    a = F.run(s, R=3, M=4, T=[1.0], seed=5, dtype="c128")
    b = oracle.ftlm(osys(w), R=3, M=4, T=np.array([1.0]), seed=5)
    assert np.abs(a["p"] - b["p"]).max() < 1e-12 * np.abs(b["p"]).max()
    s.close()
