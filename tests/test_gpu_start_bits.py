"""GPU: complex64 start vectors are the FP64 Gaussians rounded to FP32 and scaled --
the same bits as rounding numpy's FP64 values of the same stream.

numpy's log, cos and sin may differ from CUDA's in the last of 53 bits, which
changes the rounding to 24 bits of at most one value in 10^7: none is expected
among 2^20, one is allowed.  The scale is one FP32 number a vector, 1/norm to
within its last bit."""
import numpy as np
import pytest

import ftlm_workloads as W
import paper_2607_25585_gb300 as F
from gpu_helpers import empty_dev

pytestmark = pytest.mark.gpu


def philox(v, seed, dim):
    """Philox4x32-10 of counters (nu, v), nu = 0 .. dim - 1."""
    mask, u = np.uint64(0xFFFFFFFF), np.uint64
    nu = np.arange(dim, dtype=np.uint64)
    c = [nu, nu >> u(32), np.full(dim, v & 0xFFFFFFFF, np.uint64), np.full(dim, v >> 32, np.uint64)]
    k = [seed & 0xFFFFFFFF, seed >> 32]
    for _ in range(10):
        p0, p1 = c[0] * u(0xD2511F53), c[2] * u(0xCD9E8D57)
        c = [(p1 >> u(32)) ^ c[1] ^ u(k[0]), p1 & mask, (p0 >> u(32)) ^ c[3] ^ u(k[1]), p0 & mask]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return c


def gaussians(seed, v, dim):
    """rho cos and rho sin of random vector v in FP64, the turn reduced exactly."""
    c = philox(v, seed, dim)
    k1, k2 = (((c[a] << np.uint64(21)) | (c[a + 1] >> np.uint64(11))).astype(np.int64) + 1 for a in (0, 2))
    rho = np.sqrt(-2.0 * np.log(k1 * 2.0 ** -53))
    quad = (k2 + (1 << 50)) >> 51
    t = 2 * np.pi * ((k2 - (quad << 51)) * 2.0 ** -53)
    cs, sn = np.cos(t), np.sin(t)
    q = quad & 3
    return np.stack([rho * np.choose(q, [cs, -sn, -cs, sn]), rho * np.choose(q, [sn, cs, -sn, -cs])])


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("seed,off", [(0, 0), (2 ** 63 + 11, 2 ** 33 + 4)])
def test_bits_of_the_rounded_gaussians(seed, off, pairs):
    w = W.square_lattice(6, 3, seed=1)
    s = F.System.from_dict(w)
    x = empty_dev((s.dim, 2), "c64")
    (F.start_pairs if pairs else F.start_block)(s, x, 2, seed, vec_offset=off, dtype="c64")
    x = x.cpu().numpy()
    for k in range(2):
        if pairs and k:         # time reversal moves and negates, but rounds nothing
            a, b = (np.sort(np.abs(t.view(np.float32).reshape(-1))) for t in (np.ascontiguousarray(x[:, k]), np.ascontiguousarray(x[:, 0])))
            assert np.array_equal(a, b)
            continue
        z = gaussians(seed, off // 2 if pairs else off + k, s.dim).astype(np.float32)
        scale = np.float32(1.0 / np.sqrt((z.astype(np.float64) ** 2).sum()))
        wrong = [int((z * c != np.stack([x[:, k].real, x[:, k].imag])).sum())
                 for c in (scale, np.nextafter(scale, np.float32(0)), np.nextafter(scale, np.float32(1)))]
        assert min(wrong) <= 1, wrong
    s.close()
