"""GPU: what the library does when device memory runs out."""
import numpy as np
import pytest

import ftlm_workloads as W
import paper_2607_25585_gb300 as F
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu
T = np.array([0.5, 5.0])


def test_a_failed_allocation_leaves_no_error_behind():
    """A run that cannot hold its Lanczos vectors says so once; the caller's next CUDA
    call does not report it again."""
    torch = torch_cuda()
    s = F.System.from_dict(W.square_lattice(4, 4, seed=4))
    with pytest.raises(F.FtlmError) as e:      # 2^16 x 64 x 8 x 100000 bytes
        F.run(s, R=64, M=100000, T=T, seed=1, dtype="c64", symmetric=True)
    assert e.value.status == 2
    x = torch.zeros(1 << 20, device="cuda")
    x += 1
    assert float(x.sum()) == 1 << 20
    s.close()


def used():
    torch = torch_cuda()
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_a_batch_on_the_gathers_writes_no_rows():
    """Rows are written for every system of a batch or for none: 0.9 GB of the smaller
    one's would be of no use beside a sibling whose rows are too large."""
    small, large = F.System.from_dict(W.chain(11, Bdir=(1, 0, 1))), F.System.from_dict(W.chain(12, Bdir=(1, 0, 1)))
    before = used()
    F.run_batch([small, large], R=2, M=4, T=T, seed=1, dtype="c128")
    assert used() - before < 400 << 20          # workspaces: four blocks of 2 x 708,588 values, 0.1 GB
    small.close()
    large.close()


def test_rotated_blocks_are_bounded_and_shared():
    """Runs and products of one system use the same intermediate blocks, of at most 8 GB:
    22 sites, 64 vectors, three directions would be 6.4 GB for each."""
    torch = torch_cuda()
    s = F.System.from_dict(W.square_lattice(11, 2, seed=2))
    R = 64
    x = torch.view_as_complex(torch.randn(s.dim, R, 2, device="cuda"))
    y = torch.empty_like(x)
    block = s.dim * R * 8
    before = used()
    F.apply_h(s, x, y, R, "c64")                                  # two transposed blocks and the W blocks, 3 of them
    F.run(s, R=R, M=2, T=T, seed=1, dtype="c64")                  # three blocks of its own
    assert used() - before < (2 + 3 + 3) * block + (1 << 30)
    s.close()
    s = F.System.from_dict(W.square_lattice(12, 2, seed=2))       # W of 64 vectors: 25.8 GB
    before = used()
    a = F.run(s, R=R, M=3, T=T, seed=1, dtype="c64")
    assert a["shape"]["passes"] == 3 and used() - before < 3 * s.dim * R * 8 + (10 << 30)
    b = F.run(s, R=4, M=3, T=T, seed=1, vec_offset=38, dtype="c64")   # the same vectors, in one group: the same bits
    for k in ("alpha", "beta", "p"):
        assert np.array_equal(a[k][38:42], b[k])
    s.close()


def test_runs_and_products_share_their_blocks_in_order():
    """Products on two streams between runs of the same system: the same bits as alone."""
    torch = torch_cuda()
    s = F.System.from_dict(W.square_lattice(4, 4, seed=3))
    g = torch.Generator(device="cuda").manual_seed(1)
    xs = [torch.view_as_complex(torch.randn(s.dim, R, 2, device="cuda", generator=g)) for R in (3, 9, 1, 40)]
    kw = dict(R=5, M=6, T=T, seed=1, dtype="c64")
    want = []
    for x in xs:
        y = torch.empty_like(x)
        F.apply_h(s, x, y, x.shape[1], "c64")
        torch.cuda.synchronize()
        want.append(y)
    run = F.run(s, **kw)
    s.close()
    s = F.System.from_dict(W.square_lattice(4, 4, seed=3))        # (the blocks grow while products are in flight)
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = [torch.empty_like(x) for x in xs]
    torch.cuda.synchronize()
    for _ in range(4):
        for k, x in enumerate(xs):
            F.apply_h(s, x, got[k], x.shape[1], "c64", stream=streams[k % 2])
        again = F.run(s, stream=streams[0], **kw)
        assert np.array_equal(run["alpha"], again["alpha"])
        torch.cuda.synchronize()
        for p, q in zip(got, want):
            assert torch.equal(p, q)
    s.close()


def test_stored_rows_of_many_systems_are_bounded():
    """Twenty systems whose rows take 0.9 GB each: 16 GB are kept, the others' runs take
    the gathers, with the same numbers (30 x 1e-12: six steps)."""
    systems = [F.System.from_dict(W.chain(11, Bdir=(0.3, -0.2, 0.9))) for _ in range(20)]
    before = used()
    out = [F.run(s, R=4, M=6, T=T, seed=1, dtype="c128") for s in systems]
    assert used() - before < (17 << 30) + (1 << 29)               # and 20 workspaces of 45 MB
    again = F.run(systems[-1], R=4, M=6, T=T, seed=1, dtype="c128")
    assert np.array_equal(out[-1]["alpha"], again["alpha"])
    for o in out[1:]:
        for k in ("alpha", "beta", "p"):
            scale = max(np.abs(out[0][k]).max(), np.abs(out[0]["beta"]).max() * (k == "alpha"))
            assert np.abs(o[k] - out[0][k]).max() < 3e-11 * scale
    for s in systems[:2]:
        s.close()
    s = F.System.from_dict(W.chain(11, Bdir=(0.3, -0.2, 0.9)))    # room again: the stored rows' bits
    new = F.run(s, R=4, M=6, T=T, seed=1, dtype="c128")
    assert np.array_equal(new["alpha"], out[0]["alpha"])
    for t in systems[2:] + [s]:
        t.close()
    assert used() - before < 1 << 30


def test_a_stored_matrix_gives_its_memory_back():
    s = F.System.from_dict(W.square_lattice(5, 3, seed=1))
    F.CsrMatrix(s, "c64").close()
    before = used()
    for _ in range(3):
        m = F.CsrMatrix(s, "c64")
        assert used() - before > m.bytes // 2
        m.close()
        assert used() == before
    s.close()


def leave(nbytes):
    """Takes all device memory but nbytes (to 2 MB pages); nothing of it is written."""
    torch = torch_cuda()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(max(0, free - nbytes) & ~((1 << 21) - 1), dtype=torch.uint8, device="cuda")


def test_a_symmetric_run_that_fits_without_the_rotated_blocks():
    """Lanczos vectors and u.S of them come before the blocks that only make the run
    faster: 2^20 states, 64 vectors, 3 steps are 0.5 GB for each of three blocks and
    1.5 GB for each of the two; the rotated blocks would take 1.6 GB more."""
    s = F.System.from_dict(W.square_lattice(5, 4, seed=2))
    kw = dict(R=64, M=3, T=T, seed=1, dtype="c64", symmetric=True)
    hold = leave(5_400_000_000)
    a = F.run(s, **kw)
    del hold
    torch_cuda().cuda.empty_cache()
    s.close()
    s = F.System.from_dict(W.square_lattice(5, 4, seed=2))
    b = F.run(s, **kw)
    assert a["shape"]["passes"] == 1 and b["shape"]["passes"] == 3
    for k in ("alpha", "beta", "p", "M_B_sym"):         # (two gathers' roundings over three steps)
        assert np.abs(a[k] - b[k]).max() < 2e-5 * max(np.abs(b[k]).max(), np.abs(b["beta"]).max() * (k == "alpha"))
    s.close()


def test_blocks_kept_for_speed_are_given_back():
    """A run on a system whose workspace does not fit beside the rotated blocks and rows
    that other systems keep: these give way, and are made again when they are used."""
    torch = torch_cuda()
    one = F.System.from_dict(W.square_lattice(5, 4, seed=2))
    two = F.System.from_dict(W.chain(11, Bdir=(0.3, -0.2, 0.9)))
    kw1, kw2 = dict(R=64, M=3, T=T, seed=1, dtype="c64"), dict(R=4, M=3, T=T, seed=1, dtype="c128")
    a1, a2 = F.run(one, **kw1), F.run(two, **kw2)       # 1.6 GB of rotated blocks, 0.9 GB of rows
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.view_as_complex(torch.randn(two.dim, 4, 2, device="cuda", generator=g)).to(torch.complex128)
    y, z = torch.empty_like(x), torch.empty_like(x)
    F.apply_h(two, x, y, 4, "c128")                     # in flight when its rows give way
    three = F.System.from_dict(W.square_lattice(5, 4, seed=7))
    hold = leave(1_000_000_000)
    a3 = F.run(three, **kw1)                            # 1.5 GB of workspace
    del hold
    torch.cuda.empty_cache()
    assert np.isfinite(a3["lnZ"]).all()
    b1, b2 = F.run(one, **kw1), F.run(two, **kw2)
    F.apply_h(two, x, z, 4, "c128")
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    assert b1["shape"]["passes"] == 3
    for k in ("alpha", "beta", "p"):
        assert np.array_equal(a1[k], b1[k]) and np.array_equal(a2[k], b2[k])
    for s in (one, two, three):
        s.close()


def test_what_does_not_fit_is_still_refused():
    """Too little memory with nothing to give back: the same error, and the system stays usable."""
    s = F.System.from_dict(W.square_lattice(5, 4, seed=2))
    hold = leave(600_000_000)
    with pytest.raises(F.FtlmError) as e:
        F.run(s, R=64, M=3, T=T, seed=1, dtype="c64")
    assert e.value.status == 2
    del hold
    torch_cuda().cuda.empty_cache()
    assert np.isfinite(F.run(s, R=64, M=3, T=T, seed=1, dtype="c64")["lnZ"]).all()
    s.close()
