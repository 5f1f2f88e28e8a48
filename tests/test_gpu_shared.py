"""GPU: what a system's calls share -- tables written by one call and read by
another on a different stream or from another host thread."""
import threading
import time

import numpy as np
import pytest

import ftlm_workloads as W
import oracle
import paper_2607_25585_gb300 as F
from gpu_helpers import osys, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu
T = np.array([0.5, 5.0])


def dense(s, R, seed):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(s.dim, R, 2, device="cuda", generator=g))


def product(s, x, stream):
    torch = torch_cuda()
    with torch.cuda.stream(stream):           # (nothing that waits for the whole device: a run may be capturing)
        y = torch.zeros_like(x)
    F.apply_h(s, x, y, x.shape[1], "c64", stream=stream)
    stream.synchronize()
    return y


def test_product_while_the_first_run_writes_the_tables():
    """A run writes the rotated-basis tables on a stream of its own; products of one
    vector from another thread must not read them before they are there."""
    torch = torch_cuda()
    w = W.square_lattice(12, 2, seed=4)
    ref = None
    for trial in range(4):
        s = F.System.from_dict(w)
        x = dense(s, 1, 11)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        run = threading.Thread(target=F.run, args=(s,), kwargs=dict(R=1, M=2, T=T, seed=1, dtype="c64"))
        run.start()
        got = [product(s, x, stream) for _ in range(6)]
        run.join()
        ref = product(s, x, stream) if ref is None else ref
        for y in got:
            assert torch.equal(y, ref), trial
        s.close()


def test_product_after_a_run_that_failed_before_its_end():
    """A run that cannot hold its Lanczos vectors returns early; what it had begun to
    write is complete for the next product, on any stream."""
    torch = torch_cuda()
    w = W.square_lattice(12, 2, seed=4)
    s = F.System.from_dict(w)
    ref = product(s, dense(s, 1, 11), torch.cuda.Stream())
    s.close()
    s = F.System.from_dict(w)
    x = dense(s, 1, 11)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with pytest.raises(F.FtlmError) as e:      # 2^24 x 8 x 100000 bytes of them
        F.run(s, R=1, M=100000, T=T, seed=1, dtype="c64", symmetric=True)
    assert e.value.status == 2
    assert torch.equal(product(s, x, stream), ref)
    s.close()


def test_first_product_while_a_run_is_captured():
    """The rows of a small system are written by the first call that wants them; a run
    of another precision that another thread is capturing at that moment takes no
    part in it."""
    torch = torch_cuda()
    w = W.ring(N=6, two_s=2)
    kw = dict(R=2, M=150, T=T, seed=1, dtype="c64", reorth=True)     # (the row-major gather; a long capture)
    want = want_run = None
    for trial in range(12):
        s = F.System.from_dict(w)
        x = dense(s, 3, 11).to(torch.complex128)
        y = torch.zeros_like(x)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        out = {}
        run = threading.Thread(target=lambda: out.update(F.run(s, **kw)))
        run.start()
        time.sleep(0.002 * (trial % 6))
        F.apply_h(s, x, y, 3, "c128", stream=stream)
        stream.synchronize()
        run.join()
        want, want_run = (y, out) if want is None else (want, want_run)
        assert torch.equal(y, want), trial
        for k in ("alpha", "beta", "p", "lnZ"):
            assert np.array_equal(out[k], want_run[k]), (trial, k)
        s.close()
    s = F.System.from_dict(w)
    z = torch.zeros_like(want)
    F.apply_h(s, dense(s, 3, 11).to(torch.complex128), z, 3, "c128")
    torch.cuda.synchronize()
    assert torch.equal(z, want)
    s.close()


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("nvec", [1, 4])
@pytest.mark.parametrize("system", ["halves", "ones"])
def test_captured_product_leaves_the_system_usable(system, nvec, warm):
    """A product on a capturing stream takes nothing of the system's blocks, tables and
    events, whether earlier calls have made them or not: it replays, and products
    and runs after it work.  (200 roundings: 1e-6 of the norm.)"""
    torch = torch_cuda()
    w = W.square_lattice(4, 4, seed=3) if system == "halves" else W.chain(10, Bdir=(0.3, -0.2, 0.9))
    s = F.System.from_dict(w)
    x = dense(s, nvec, 5)
    ref = oracle.apply_h(osys(w), x.cpu().numpy().astype(np.complex128))
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    if warm:
        F.apply_h(s, x, y, nvec, "c64")
        F.run(s, R=nvec, M=3, T=T, seed=1, dtype="c64")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        F.apply_h(s, x, y, nvec, "c64")
    y.zero_()
    z = torch.zeros_like(x)
    F.apply_h(s, x, z, nvec, "c64")           # before the graph has ever run
    torch.cuda.synchronize()
    assert rel_l2(z.cpu().numpy(), ref) < 1e-6
    a = F.run(s, R=nvec, M=3, T=T, seed=1, dtype="c64")
    g.replay()
    torch.cuda.synchronize()
    assert rel_l2(y.cpu().numpy(), ref) < 1e-6
    b = F.run(s, R=nvec, M=3, T=T, seed=1, dtype="c64")
    assert np.array_equal(a["alpha"], b["alpha"])
    s.close()


@pytest.mark.parametrize("system", ["halves", "ones", "small ones"])
def test_first_products_while_another_thread_captures(system):
    """A system's first products allocate and write what they keep; a capture that
    another thread has open (in CUDA's default, global mode) and the products both
    come to their end."""
    torch = torch_cuda()
    w = {"halves": lambda: W.square_lattice(4, 4, seed=3), "ones": lambda: W.chain(10, Bdir=(0.3, -0.2, 0.9)),
         "small ones": lambda: W.chain(7, Bdir=(0.3, -0.2, 0.9))}[system]()
    s = F.System.from_dict(w)
    blocks = [dense(s, nvec, 5) for nvec in (4, 1)]
    outs = [torch.zeros_like(x) for x in blocks]
    a = torch.ones(1 << 10, device="cuda")
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    fault = []

    def products():
        try:
            for x, y in zip(blocks, outs):
                F.apply_h(s, x, y, x.shape[1], "c64", stream=other)
        except Exception as e:  # noqa: BLE001 (told to the test's thread)
            fault.append(e)

    with torch.cuda.graph(g, stream=stream):
        a.add_(1)
        t = threading.Thread(target=products)
        t.start()
        t.join()
        a.mul_(2)
    assert not fault
    g.replay()
    torch.cuda.synchronize()
    assert float(a[0]) == 4.0
    for x, y in zip(blocks, outs):
        ref = oracle.apply_h(osys(w), x.cpu().numpy().astype(np.complex128))
        assert rel_l2(y.cpu().numpy(), ref) < 1e-6
    s.close()


def test_systems_come_and_go_while_others_capture():
    """Eight threads that create a system, run it and destroy it: what waits for the
    whole device (a destruction) waits for the captures of other threads' runs too."""
    w = W.ring(N=6, two_s=2)
    kw = dict(R=2, M=120, T=T, dtype="c64", reorth=True)     # (a long capture)
    s = F.System.from_dict(w)
    want = F.run(s, seed=1, **kw)
    s.close()
    faults = []

    def work():
        for _ in range(6):
            try:
                s = F.System.from_dict(w)
                r = F.run(s, seed=1, **kw)
                s.close()
                if not np.array_equal(r["alpha"], want["alpha"]):
                    faults.append("other numbers")
            except Exception as e:  # noqa: BLE001 (told to the test's thread)
                faults.append(e)

    threads = [threading.Thread(target=work) for _ in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults[:3]


def test_more_runs_at_once_than_captured_runs_are_kept():
    """Eleven threads, each with a system and runs of its own: a run's captured graph
    stays until the run has ended, however many others are captured meanwhile."""
    w = W.ring(N=6, two_s=2)
    T40 = np.geomspace(1, 50, 40)
    kw = dict(R=24, M=60, T=T40, dtype="c128")

    def work(k, out):
        s = F.System.from_dict(w)
        out[k] = [F.run(s, seed=100 * k + j, **kw) for j in range(4)]
        s.close()

    alone, at_once = {}, {}
    for k in range(11):
        work(k, alone)
    threads = [threading.Thread(target=work, args=(k, at_once)) for k in range(11)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(11):
        for a, b in zip(alone[k], at_once[k]):
            for q in ("alpha", "beta", "p", "lnZ", "M_B"):
                assert np.array_equal(a[q], b[q]), (k, q)
