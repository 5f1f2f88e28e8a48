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
