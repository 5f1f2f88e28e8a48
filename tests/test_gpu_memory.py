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
