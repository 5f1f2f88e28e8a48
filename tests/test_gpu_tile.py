"""GPU: the tile gather (complex64, general spins, d >= 2^15) against the forced
row-major kernel and the register-cube gather: top spins 1/2 to 5/2, group
remainders, low tiles from 125 to 256 bases, mixed radices, batches.

Tolerances: a row adds at most 250 products, 30 units roundoff of the sum of
magnitudes: 2e-6 of the norm for a product; six steps amplify it by less than
ten."""
import numpy as np
import pytest
from conftest import random_system

import ftlm_workloads as W
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev, rel_l2, to_dev

pytestmark = pytest.mark.gpu
T = np.array([1.0, 10.0])
SYSTEMS = {
    "ones": [2] * 10,                        # 3^10, tile 243
    "threehalves": [3] * 8,                  # 4^8, tile 256
    "twos": [4] * 7,                         # 5^7, tile 125
    "cube": [5] + [4] * 6,                   # 6 * 5^6, tile 150
    "halves on ones": [2] * 9 + [1, 1],      # top spin 1/2
    "mixed": [3, 1, 2, 5, 1, 2, 2, 3, 5],    # 4 2 3 6 2 3 3 4 6
    "fives": [5] * 6,                        # 6^6, tile 216
}


@pytest.mark.parametrize("name", SYSTEMS)
@pytest.mark.parametrize("R", [2, 3, 5, 8])
def test_tile_gather(name, R, rng):
    s = F.System.from_dict(random_system(np.random.default_rng(11), SYSTEMS[name]))
    assert s.dim >= 2 ** 15
    x = to_dev(rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R)), "c64")
    y, z = empty_dev((s.dim, R), "c64"), empty_dev((s.dim, R), "c64")
    F.apply_h(s, x, y, R, "c64")
    a = F.run(s, R=R, M=6, T=T, seed=2, dtype="c64")
    assert a["shape"]["site_cube"] == SYSTEMS[name][-1] + 1 and a["shape"]["vector_major"] == 1
    F.tune_shape(s, R, "c64", 0, 1, 1, 0)    # the row-major general kernel
    try:
        F.apply_h(s, x, z, R, "c64")
        b = F.run(s, R=R, M=6, T=T, seed=2, dtype="c64")
    finally:
        F.tune_shape(s, R, "c64", -1)
    assert rel_l2(y.cpu().numpy(), z.cpu().numpy()) < 2e-6
    scale = np.abs(b["beta"]).max()
    for k in ("alpha", "beta"):
        assert np.abs(a[k] - b[k]).max() < 2e-5 * max(scale, np.abs(b["alpha"]).max())
    assert np.abs(a["p"] - b["p"]).max() < 2e-5 * np.abs(b["p"]).max()
    s.close()


def test_tile_batch_matches_single_runs():
    """Systems of one low tile and different lengths, groups that end inside a system."""
    ss = [F.System.from_dict(W.chain(n, Bdir=(0.3, 0.2, 0.9))) for n in (10, 11, 10)]
    rs = F.run_batch(ss, R=6, M=5, T=T, seed=4, dtype="c64")
    for s, r in zip(ss, rs):
        one = F.run(s, R=6, M=5, T=T, seed=4, dtype="c64")
        assert r["shape"]["site_cube"] == 3 and r["shape"]["group_vectors"] == 4
        for k in ("alpha", "beta", "p"):
            assert np.abs(r[k] - one[k]).max() < 2e-6 * max(np.abs(one[k]).max(), np.abs(one["beta"]).max() * (k == "alpha"))
        s.close()


@pytest.mark.parametrize("name", ["ones", "cube"])
def test_autotuned_runs(name):
    """The autotuner times the tile gather with the other shapes: whichever it keeps,
    the run's results are the default plan's, and a later product is right."""
    s = F.System.from_dict(random_system(np.random.default_rng(12), SYSTEMS[name]))
    kw = dict(R=4, M=6, T=T, seed=2, dtype="c64")
    a, b = F.run(s, **kw), F.run(s, autotune=True, **kw)
    x, y, z = (empty_dev((s.dim, 4), "c64") for _ in range(3))
    F.start_block(s, x, 4, 2, dtype="c64")
    F.apply_h(s, x, y, 4, "c64")
    F.tune_shape(s, 4, "c64", -1)
    F.apply_h(s, x, z, 4, "c64")
    assert rel_l2(y.cpu().numpy(), z.cpu().numpy()) < 2e-6
    scale = max(np.abs(b["beta"]).max(), np.abs(b["alpha"]).max())
    for k in ("alpha", "beta"):
        assert np.abs(a[k] - b[k]).max() < 2e-5 * scale
    s.close()
