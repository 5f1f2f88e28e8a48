"""GPU: the rotated-basis H.v of spin-1/2 runs (random and time-reversed-pair
starts) against the oracle and against the gather, which the same run takes
from a caller's block of the same start vectors.

Tolerances: a step rounds about 100 times a value, so its relative error is
about 10 units roundoff (6e-8 / 1.1e-16); eight steps that have not lost
orthogonality amplify it by less than 30: 2e-5 in complex64, 1e-13 (with the
oracle's own error 1e-12) in complex128, relative to the largest coefficient."""
import numpy as np
import pytest

import ftlm_workloads as W
import oracle
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev, osys, to_dev

pytestmark = pytest.mark.gpu
T = np.array([0.5, 2.0, 20.0])


def close(a, b, tol):
    for k in ("alpha", "beta", "p"):
        scale = np.abs(b["alpha"]).max() if k == "alpha" else np.abs(b[k]).max()
        scale = max(scale, np.abs(b["beta"]).max()) if k == "alpha" else scale
        assert np.abs(a[k] - b[k]).max() < tol * scale, k
    assert list(a["M_eff"]) == list(b["M_eff"])


def buckled(lx, ly):
    w = W.square_lattice(lx, ly, seed=5, B=1.3, Bdir=(0.3, -0.5, 0.8))
    w["pos"][:, 2] = 0.5 * np.cos(1.3 * np.arange(lx * ly))
    return w


SYSTEMS = {
    "chain13": lambda: W.square_lattice(13, 1, seed=1, Bdir=(1, 2, 3)),      # x, y and z: one low tile pair
    "lattice14": lambda: W.square_lattice(7, 2, seed=2, Bdir=(0, 0, 1)),     # three directions in the plane
    "buckled15": lambda: buckled(5, 3),                                      # five directions
    "ladder16": lambda: W.ladder(8, dipolar=False),                          # exchange alone
    "buckled16": lambda: buckled(4, 4),
    "ring13": lambda: W.ring(13, two_s=1, radius=5.0, Bdir=(1, 2, 2)),       # bonds at every angle of the plane
    "ring15": lambda: W.ring(15, two_s=1, radius=6.0),
}


@pytest.mark.parametrize("name", SYSTEMS)
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_rotated_run_matches_oracle(name, dtype):
    w = SYSTEMS[name]()
    s = F.System.from_dict(w)
    for R, start in ((3, "random"), (2, "pairs")):
        g = F.run(s, R=R, M=8, T=T, seed=7, vec_offset=2, start=start, dtype=dtype)
        assert g["shape"]["passes"] == 3 and g["shape"]["vector_major"] == 1
        x = empty_dev((s.dim, R), dtype)
        (F.start_pairs if start == "pairs" else F.start_block)(s, x, R, 7, vec_offset=2, dtype=dtype)
        close(g, F.run(s, R=R, M=8, T=T, start="user", user_start=x, dtype=dtype), 2e-5 if dtype == "c64" else 1e-12)
        if start == "random":
            close(g, oracle.ftlm(osys(w), R=R, M=8, T=T, seed=7, vec_offset=2), 2e-5 if dtype == "c64" else 1e-12)
    s.close()


@pytest.mark.parametrize("n", [17, 18, 19, 20, 21, 22, 23, 24, 25])
def test_rotated_run_matches_gather_at_every_split(n):
    """Every split of the index into tile and column bits, on both sides of the
    change of tile size."""
    w = W.square_lattice(n, 1, seed=n, Bdir=(1, 1, 0))
    s = F.System.from_dict(w)
    for dtype, tol in (("c64", 2e-5), ("c128", 1e-12)):
        if dtype == "c128" and n > 23:
            continue
        R = 2 if n < 23 else 1
        g = F.run(s, R=R, M=3, T=T, seed=3, dtype=dtype)
        assert g["shape"]["passes"] == 3
        x = empty_dev((s.dim, R), dtype)
        F.start_block(s, x, R, 3, dtype=dtype)
        close(g, F.run(s, R=R, M=3, T=T, start="user", user_start=x, dtype=dtype), tol)
    s.close()


@pytest.mark.parametrize("n,R", [(24, 3), (26, 2), (27, 1)])
def test_large_middle_tiles(n, R):
    """The middle pass over its large tile: a CTA takes several tiles in turn, of one
    vector or more, and with few enough columns every group of the index has high bits."""
    w = W.square_lattice(n, 1, seed=n, Bdir=(1, 1, 0))
    s = F.System.from_dict(w)
    g = F.run(s, R=R, M=3, T=T, seed=3, dtype="c64")
    assert g["shape"]["passes"] == 3
    x = empty_dev((s.dim, R), "c64")
    F.start_block(s, x, R, 3, dtype="c64")
    close(g, F.run(s, R=R, M=3, T=T, start="user", user_start=x, dtype="c64"), 2e-5)
    s.close()


def test_starts_that_may_be_sparse_keep_the_gather():
    """An isotropic system conserves S^z: from a basis state the run stays in its
    sector and ends where the sector ends."""
    n = 13
    J = np.zeros((n, n))
    J[0, 1] = 1.0
    s = F.System([1] * n, J=J, B=[0, 0, 0.3])
    g = F.run(s, R=1, M=6, T=T, start="basis", basis_offset=1, dtype="c64")
    assert g["shape"]["passes"] == 1 and list(g["M_eff"]) == [2]
    s.close()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("R", [1, 3, 4])
def test_product_on_dense_and_other_blocks(R, dtype, rng):
    """ftlm_apply_h: a dense block (rotated passes), and blocks with one vector
    that is not (the gather): a basis state, whose product is exactly zero where H
    has no element; a value that is not finite, which reaches only its
    neighbours; values near the ends of the range.  Tolerance of a product:
    about 200 roundings, 15 units roundoff, relative to the norm."""
    w = buckled(4, 4)
    s = F.System.from_dict(w)
    tol = 1e-6 if dtype == "c64" else 4e-15 + 1e-13
    x = rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R))

    def product(x):
        y = empty_dev((s.dim, R), dtype)
        xd = to_dev(x, dtype)
        F.apply_h(s, xd, y, R, dtype)
        return xd.cpu().numpy().astype(np.complex128), y.cpu().numpy()

    def check(x, y, cols):
        ref = oracle.apply_h(osys(w), np.ascontiguousarray(x[:, cols]))
        for k, c in enumerate(cols):
            top = np.abs(ref[:, k]).max()     # (a norm's squares may leave the range)
            assert np.linalg.norm((y[:, c] - ref[:, k]) / top) < tol * np.linalg.norm(ref[:, k] / top)
        return ref

    check(*product(x), range(R))
    e = x.copy()
    e[:, R - 1] = 0
    e[777, R - 1] = 1
    xe, y = product(e)
    ref = check(xe, y, range(R))
    assert np.all(y[ref[:, -1] == 0, R - 1] == 0)
    for scale in ((1e-30, 1e28) if dtype == "c64" else (1e-200, 1e200)):
        check(*product(x * scale), range(R))
    bad = x.copy()
    bad[777, R - 1] = np.nan
    y = product(bad)[1]
    assert np.array_equal(np.isnan(y[:, R - 1].real), np.abs(ref[:, -1]) > 0)
    s.close()


def test_products_on_two_streams():
    """Two products of one system on different streams share its blocks in order."""
    torch = pytest.importorskip("torch")
    w = W.square_lattice(4, 4, seed=3)
    s = F.System.from_dict(w)
    g = torch.Generator(device="cuda").manual_seed(1)
    xs = [torch.view_as_complex(torch.randn(s.dim, R, 2, device="cuda", generator=g)) for R in (8, 5, 1, 8)]
    want = []
    for x in xs:
        y = torch.empty_like(x)
        F.apply_h(s, x, y, x.shape[1], "c64")
        torch.cuda.synchronize()
        want.append(y)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    got = [torch.empty_like(x) for x in xs]
    torch.cuda.synchronize()
    for _ in range(3):
        for k, x in enumerate(xs):
            F.apply_h(s, x, got[k], x.shape[1], "c64", stream=(a, b)[k % 2])
    torch.cuda.synchronize()
    for p, q in zip(got, want):
        assert torch.equal(p, q)
    s.close()


@pytest.mark.parametrize("name", ["buckled", "lattice", "ladder"])
def test_product_has_no_systematic_error(name):
    """The part of a complex64 product's error that lies along the exact product, on
    a dense block of 20 sites with five, three and two directions.  Roundings of
    single values are independent and leave 6e-8 / sqrt(2^20) of it; what remains
    is a factor common to all values (the gates', the tables' scale), which has to
    be below one unit roundoff."""
    torch = pytest.importorskip("torch")
    w = {"buckled": lambda: buckled(4, 5), "lattice": lambda: W.square_lattice(4, 5, seed=2),
         "ladder": lambda: W.ladder(10, dipolar=False)}[name]()
    s = F.System.from_dict(w)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.view_as_complex(torch.randn(s.dim, 2, 2, device="cuda", generator=g))
    y, ref = torch.empty_like(x), empty_dev(x.shape, "c128")
    F.apply_h(s, x, y, 2, "c64")
    F.apply_h(s, x.to(torch.complex128), ref, 2, "c128")
    torch.cuda.synchronize()
    for k in range(2):
        along = torch.vdot(ref[:, k], y[:, k] - ref[:, k]).real / torch.vdot(ref[:, k], ref[:, k]).real
        assert abs(float(along)) < 2.0 ** -24
    s.close()


def sectors(n):
    mu = np.arange(1 << n)
    return np.array([bin(m).count("1") for m in mu])


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("R", [1, 3])
def test_sectors_without_weight_stay_without_weight(dtype, R, rng):
    """A Hamiltonian that conserves S^z and a block whose outer sectors are exactly
    zero -- two rows of them, or a few hundred -- in its last vector: so is the product."""
    w = W.ladder(8, dipolar=False)
    s = F.System.from_dict(w)
    up = sectors(16)
    for keep in (1, 3):
        x = rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R))
        out = (up < keep) | (up > 16 - keep)
        x[out, -1] = 0
        y = empty_dev((s.dim, R), dtype)
        F.apply_h(s, to_dev(x, dtype), y, R, dtype)
        y = y.cpu().numpy()
        assert np.all(y[out, -1] == 0) and np.all(y[~out, -1] != 0), keep
    s.close()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("amplitude", [2.0 ** -46, 2.0 ** -20, 2.0 ** -12, 2.0 ** -8])
def test_small_sectors_keep_their_digits(dtype, amplitude, rng):
    """The same with one sector of 1820 rows (1 in 36) at a small amplitude: its rows of
    the product have the error of their own terms (200 roundings, 15 units roundoff
    of the sector's norm), not of the vector's."""
    w = W.ladder(8, dipolar=False)
    s = F.System.from_dict(w)
    x = rng.normal(size=(s.dim, 2)) + 1j * rng.normal(size=(s.dim, 2))
    small = sectors(16) == 4
    x[small, 1] *= amplitude
    xd = to_dev(x, dtype)
    y = empty_dev((s.dim, 2), dtype)
    F.apply_h(s, xd, y, 2, dtype)
    ref = oracle.apply_h(osys(w), xd.cpu().numpy().astype(np.complex128))
    tol = 1e-6 if dtype == "c64" else 4e-15 + 1e-13
    e = y.cpu().numpy() - ref
    for rows in (small, ~small):
        for k in range(2):
            assert np.linalg.norm(e[rows, k]) < tol * np.linalg.norm(ref[rows, k])
    s.close()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_vectors_of_a_block_do_not_choose_for_each_other(dtype, rng):
    """A vector's product has the same bits whichever vectors share its block."""
    w = buckled(4, 4)
    s = F.System.from_dict(w)
    R = 5
    x = rng.normal(size=(s.dim, R)) + 1j * rng.normal(size=(s.dim, R))
    y = [empty_dev((s.dim, R), dtype) for _ in range(3)]
    F.apply_h(s, to_dev(x, dtype), y[0], R, dtype)
    x[:, 1] = 0
    x[4321, 1] = 1
    F.apply_h(s, to_dev(x, dtype), y[1], R, dtype)
    x[:, [0, 2, 3, 4]] = x[:, [1, 1, 1, 1]]
    F.apply_h(s, to_dev(x, dtype), y[2], R, dtype)
    a, b, c = (t.cpu().numpy() for t in y)
    for k in (0, 2, 3, 4):
        assert np.array_equal(a[:, k], b[:, k]) and np.array_equal(c[:, k], b[:, 1])
    s.close()


@pytest.mark.parametrize("dtype,shape,flat", [("c64", (5, 5), False), ("c64", (13, 2), False), ("c64", (7, 4), True),
                                              ("c128", (12, 2), True), ("c128", (5, 5), False), ("c128", (13, 2), False)])
def test_largest_tiles_and_five_directions(dtype, shape, flat):
    """The large tiles with three and five directions, the largest systems of either
    precision: the run against the gather's from the same start vector."""
    w = W.square_lattice(*shape, seed=3, Bdir=(1, 1, 0)) if flat else buckled(*shape)
    s = F.System.from_dict(w)
    g = F.run(s, R=1, M=3, T=T, seed=3, dtype=dtype)
    assert g["shape"]["passes"] == 3
    x = empty_dev((s.dim, 1), dtype)
    F.start_block(s, x, 1, 3, dtype=dtype)
    close(g, F.run(s, R=1, M=3, T=T, start="user", user_start=x, dtype=dtype), 2e-5 if dtype == "c64" else 1e-12)
    s.close()
