"""GPU: complex64 start vectors (two-float Box-Muller) against the complex128
ones (FP64 log and sincospi) of the same stream.

Tolerance: a complex64 value is the Gaussian rounded to FP32 (1.02 * 2^-24 with
the two-float form's own error), times the scale rounded to FP32 (2^-24), the
product rounded (2^-24), against the FP64 value: 3.1 * 2^-24 relative, value by
value and part by part."""
import numpy as np
import pytest

import ftlm_workloads as W
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 3, 8])
@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("system", ["ring", "lattice"])
def test_complex64_start_is_the_rounded_complex128_start(system, pairs, R):
    s = F.System.from_dict(W.ring(N=9, two_s=2) if system == "ring" else W.square_lattice(4, 4, seed=1))
    start = F.start_pairs if pairs else F.start_block
    a, b = empty_dev((s.dim, R), "c64"), empty_dev((s.dim, R), "c128")
    for seed, off in ((0, 0), (2 ** 63 + 11, 2 ** 33 + 5)):
        start(s, a, R, seed, vec_offset=off, dtype="c64")
        start(s, b, R, seed, vec_offset=off, dtype="c128")
        x, y = a.cpu().numpy().astype(np.complex128), b.cpu().numpy()
        for p, q in ((x.real, y.real), (x.imag, y.imag)):
            assert np.all(np.abs(p - q) <= 3.1 * 2.0 ** -24 * np.abs(q))
    s.close()
