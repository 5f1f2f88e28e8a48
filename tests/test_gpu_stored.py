"""GPU: products and steps of small systems from stored rows, against the oracle
and the forced gathers: group sizes and remainders, rows that are no multiple of
a CTA's 32, exact zeros, calls inside a stream capture.

Tolerances: a row adds at most 200 products in two levels, so its relative
error is below 30 units roundoff of the sum of magnitudes; the norms used here
give 2e-6 in complex64 and 4e-15 in complex128 (1e-12 with the oracle's)."""
import numpy as np
import pytest
from conftest import random_system

import ftlm_workloads as W
import oracle
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev, osys, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu
TOL = {"c64": 2e-6, "c128": 1e-12}
SYSTEMS = {
    "one site": [4],
    "two halves": [1, 1],
    "mixed": [1, 2, 3, 5, 1, 2],
    "halves": [1] * 11,
    "ones": [2] * 6,
    "large spins": [15, 7, 3],
}


@pytest.mark.parametrize("name", SYSTEMS)
@pytest.mark.parametrize("R", [1, 2, 3, 4, 7, 8])
def test_stored_product_matches_oracle(name, R, rng):
    w = random_system(np.random.default_rng(5), SYSTEMS[name])
    s = F.System.from_dict(w)
    x = rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R))
    for dtype in ("c64", "c128"):
        xd = to_dev(x, dtype)
        ref = oracle.apply_h(osys(w), xd.cpu().numpy().astype(np.complex128))
        for _ in range(2):          # the call that writes the rows, and one that finds them
            y = empty_dev((s.dim, R), dtype)
            F.apply_h(s, xd, y, R, dtype)
            assert rel_l2(y.cpu().numpy(), ref) < TOL[dtype]
    s.close()


def test_rows_that_are_not_connected_stay_zero():
    J = np.zeros((10, 10))
    J[0, 1] = J[1, 2] = 0.7
    s = F.System([1] * 10, J=J, B=(0, 0, 0.4))
    x = np.zeros((s.dim, 1))
    x[1] = 1.0                      # one spin up: H keeps their number
    y = empty_dev((s.dim, 1), "c64")
    F.apply_h(s, to_dev(x, "c64"), y, 1, "c64")
    got = y.cpu().numpy()[:, 0]
    assert set(np.flatnonzero(got)) <= {1, 2} and got[2] != 0
    s.close()


@pytest.mark.parametrize("R", [1, 6, 8])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_stored_run_matches_forced_gather(R, dtype):
    T = np.array([0.5, 5.0])
    w = W.chain(7, Bdir=(0.3, -0.2, 0.9))           # d = 2187
    s = F.System.from_dict(w)
    a = F.run(s, R=R, M=10, T=T, seed=3, dtype=dtype)
    F.tune_shape(s, R, dtype, 0, 0, 1, 1)           # the one-row vector-major gather
    try:
        b = F.run(s, R=R, M=10, T=T, seed=3, dtype=dtype)
    finally:
        F.tune_shape(s, R, dtype, -1)
    for k in ("alpha", "beta", "p"):                # ten steps amplify rounding by less than 30
        assert np.abs(a[k] - b[k]).max() < 30 * TOL[dtype] * max(np.abs(b[k]).max(), np.abs(b["beta"]).max() * (k == "alpha"))
    s.close()


def test_product_inside_a_capture():
    torch = torch_cuda()
    w = W.ring(N=5, two_s=2)
    x = torch.randn(243, 4, dtype=torch.complex128, device="cuda")
    ref = oracle.apply_h(osys(w), x.cpu().numpy())
    for warm in (False, True):      # the gather is captured, whether the rows have been written or not
        s = F.System.from_dict(w)
        y = torch.empty_like(x)
        if warm:
            F.apply_h(s, x, y, 4, "c128")
            torch.cuda.synchronize()
            F.apply_h(s, x, y, 4, "c128")
            y.zero_()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            F.apply_h(s, x, y, 4, "c128")
        g.replay()
        torch.cuda.synchronize()
        assert rel_l2(y.cpu().numpy(), ref) < 1e-12
        s.close()


@pytest.mark.parametrize("R", [1, 5, 16, 40, 80, 200])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_whole_run_in_one_launch_matches_steps(R, dtype):
    """Clusters of 8, 4, 2 and 1 CTAs a vector (by the number of vectors) against the
    same run step by step (kernel timing asks for it), for rows that the CTAs do
    not share evenly, a symmetric run's stored vectors, and a breakdown."""
    T = np.array([0.5, 5.0])
    for ts in ([2] * 5, [4], [1, 2, 1]):
        w = random_system(np.random.default_rng(8), ts)
        s = F.System.from_dict(w)
        M = min(10, s.dim + 2)
        kw = dict(R=R, M=M, T=T, seed=3, dtype=dtype, symmetric=len(ts) == 5)
        a, b = F.run(s, **kw), F.run(s, time_kernels=True, **kw)
        assert list(a["M_eff"]) == list(b["M_eff"])
        m = min(M, max(1, s.dim // 3))              # the steps well before the Krylov space is exhausted
        for k in ("alpha", "beta", "p"):
            scale = max(np.abs(b[k][:, :m]).max(), np.abs(b["beta"]).max() * (k == "alpha"))
            assert np.abs(a[k][:, :m] - b[k][:, :m]).max() < 30 * TOL[dtype] * scale, (ts, k)
        if len(ts) == 5:
            assert np.abs(a["O"] - b["O"]).max() < 30 * TOL[dtype] * np.abs(b["O"]).max()
        s.close()


@pytest.mark.parametrize("dtype,R", [("c128", 1), ("c128", 3), ("c128", 8)])
def test_rows_beyond_l2(dtype, R):
    """Complex128 systems keep their rows up to 2 GB: products and
    runs against the forced row-major gather (d = 59,049)."""
    T = np.array([0.5, 5.0])
    w = W.chain(10, Bdir=(0.3, -0.2, 0.9))
    s = F.System.from_dict(w)
    g = np.random.default_rng(4)
    x = to_dev(g.normal(size=(s.dim, R)) + 1j * g.normal(size=(s.dim, R)), dtype)
    y, z = empty_dev((s.dim, R), dtype), empty_dev((s.dim, R), dtype)
    F.apply_h(s, x, y, R, dtype)    # (one and three vectors: the gather)
    first = y.clone()
    a = F.run(s, R=R, M=6, T=T, seed=3, dtype=dtype)
    F.tune_shape(s, R, dtype, 0, 1, 1, 0)
    try:
        F.apply_h(s, x, z, R, dtype)
        b = F.run(s, R=R, M=6, T=T, seed=3, dtype=dtype)
    finally:
        F.tune_shape(s, R, dtype, -1)
    assert rel_l2(y.cpu().numpy(), z.cpu().numpy()) < TOL[dtype]
    F.apply_h(s, x, y, R, dtype)    # after a run has written the rows: the same bits
    assert bool((y == first).all())
    for k in ("alpha", "beta", "p"):
        scale = max(np.abs(b[k]).max(), np.abs(b["beta"]).max() * (k == "alpha"))
        assert np.abs(a[k] - b[k]).max() < 10 * TOL[dtype] * scale
    s.close()


@pytest.mark.parametrize("batch", [False, True])
def test_autotuned_runs_keep_their_stored_rows(batch):
    """The autotuner and the run agree on which runs take stored rows (one vector, six
    products: they do): the same bits with and without it, and no shape left behind."""
    T = np.array([0.5, 5.0])
    systems = [F.System.from_dict(W.chain(10, Bdir=d)) for d in ((0.3, -0.2, 0.9), (1, 0, 0.5))][:1 + batch]
    kw = dict(R=1, M=6, T=T, seed=3, dtype="c128")
    go = (lambda **k: F.run_batch(systems, **k)) if batch else (lambda **k: [F.run(systems[0], **k)])
    a, b, c = go(**kw), go(autotune=True, **kw), go(**kw)
    for x, y, z in zip(a, b, c):
        for k in ("alpha", "beta", "p"):
            assert np.array_equal(x[k], y[k]) and np.array_equal(x[k], z[k])
    for s in systems:
        F.tune_shape(s, 1, "c128", -1)
        s.close()


MANY = {"halves11": (lambda: W.square_lattice(11, 1, seed=1), (8, 9, 64)),
        "halves12": (lambda: W.square_lattice(12, 1, seed=1), (16, 23, 24, 130)),
        "halves14": (lambda: W.square_lattice(14, 1, seed=1), (4, 8, 9, 128)),
        "bonds14": (lambda: W.ladder(7, dipolar=False), (32, 64, 200)),
        "ones8": (lambda: W.chain(8, Bdir=(0.3, -0.2, 0.9)), (128, 200)),
        "threehalves6": (lambda: W.ring(N=6, two_s=3), (128, 256)),
        "large spins": (lambda: W.ring(N=4, two_s=9), (9, 64, 128))}


@pytest.mark.parametrize("name", MANY)
def test_products_of_many_vectors_on_both_sides_of_the_rule(name, rng):
    """Blocks that take stored rows and blocks that take the gathers, against the oracle."""
    w, sizes = MANY[name][0](), MANY[name][1]
    s = F.System.from_dict(w)
    for R in sizes:
        x = to_dev(rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R)), "c64")
        y = empty_dev((s.dim, R), "c64")
        F.apply_h(s, x, y, R, "c64")
        cols = [0, R // 2, R - 1]
        ref = oracle.apply_h(osys(w), np.ascontiguousarray(x.cpu().numpy()[:, cols]).astype(np.complex128))
        assert rel_l2(y.cpu().numpy()[:, cols], ref) < TOL["c64"]
    s.close()


def test_products_of_many_vectors_are_not_left_to_the_rows():
    """14 spins 1/2 and 128 vectors: the gathers take 0.09 ms, the stored rows 0.8 ms."""
    torch = torch_cuda()
    s = F.System.from_dict(W.square_lattice(14, 1, seed=1))
    x = torch.view_as_complex(torch.randn(s.dim, 128, 2, device="cuda"))
    y = torch.empty_like(x)
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(3):
        F.apply_h(s, x, y, 128, "c64")
    a.record()
    for _ in range(10):
        F.apply_h(s, x, y, 128, "c64")
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) / 10 < 0.3
    s.close()


def test_batches_of_small_systems_keep_their_rows():
    """The rule on entries and vectors looks at each system of a batch by itself: 24
    systems that take rows alone take them together (0.15 ms a step; the gathers
    0.56 ms).  Five steps amplify the roundings of another order by less than 30."""
    T = np.array([0.5, 5.0])
    systems = [F.System.from_dict(W.square_lattice(10, 1, seed=k, Bdir=(1, k, 2))) for k in range(24)]
    kw = dict(R=48, M=5, T=T, seed=3, dtype="c64", time_kernels=True)
    F.run_batch(systems, **kw)
    together = F.run_batch(systems, **kw)
    assert together[0]["hv_ms"] / 5 < 0.3
    for s, b in list(zip(systems, together))[::7]:
        a = F.run(s, **kw)
        for k in ("alpha", "beta", "p"):
            scale = max(np.abs(a[k]).max(), np.abs(a["beta"]).max() * (k == "alpha"))
            assert np.abs(a[k] - b[k]).max() < 30 * TOL["c64"] * scale
    for s in systems:
        s.close()
