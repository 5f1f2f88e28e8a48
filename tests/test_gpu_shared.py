"""GPU: what a system's calls share -- tables written by one call and read by
another on a different stream or from another host thread."""
import threading

import numpy as np
import pytest

import ftlm_workloads as W
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev, torch_cuda

pytestmark = pytest.mark.gpu
T = np.array([0.5, 5.0])


def dense(s, R, seed):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(s.dim, R, 2, device="cuda", generator=g))


def product(s, x, stream):
    y = empty_dev(x.shape, "c64")
    y.zero_()
    torch_cuda().cuda.synchronize()
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
