"""Quantisation over the reduced range, whose boundaries the kernel forms itself,
against quantisation over the same range given by the caller (boundaries from the
host): the same codes and codebook for every form of the kernels."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_01127_gb300 import workloads

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def logq():
    return lib()


# bases on both sides of the level estimates' limits; scales whose first boundary is
# ordinary, near the smallest normal number, subnormal, 0 or near the largest
@pytest.mark.parametrize("bits,base", [(4, 2.0), (4, 1.08), (4, 1.09), (4, 7.9), (4, 8.1), (3, 2.0), (3, 1.08), (3, 8.1),
                                       (8, 1.05), (8, 1.006), (8, 1.0071), (8, 15.9), (8, 16.1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -118, 2.0 ** -122, 2.0 ** -136, 2.0 ** 120])
@pytest.mark.parametrize("N,K", [(3, 128), (37, 1152)])
def test_reduced_range_equals_given_range(logq, bits, base, scale, N, K):
    w = workloads.weights_np(N, K, seed=N + K + bits) * np.float32(scale)
    w[0, :3] = [0.0, -0.0, np.abs(w).max()]
    W = torch.from_numpy(w).cuda()
    codes, cb = logq.logq_quantize(W, bits, base)
    want, wcb = logq.logq_quantize(W, bits, base, range_=float(np.abs(w).max()))
    assert torch.equal(codes, want)
    assert bytes(cb) == bytes(wcb)


@pytest.mark.parametrize("bits,base", [(8, 1e30), (4, 1e100), (3, 1e300)])
def test_boundaries_below_fp64(logq, bits, base):
    """Boundaries that underflow fp64 to 0: zeros keep code 0, the smallest subnormals do not."""
    w = workloads.weights_np(9, 256, seed=bits)
    w[0, :4] = [0.0, -0.0, np.nextafter(np.float32(0), np.float32(1)), -1e-40]
    W = torch.from_numpy(w).cuda()
    codes, cb = logq.logq_quantize(W, bits, base)
    want, wcb = logq.logq_quantize(W, bits, base, range_=float(np.abs(w).max()))
    assert torch.equal(codes, want) and bytes(cb) == bytes(wcb)
    m = (np.abs(w)[..., None] >= np.array(cb.thresh[:cb.qmax], np.float32)).sum(-1)
    q = oracle.unpack(codes.cpu().numpy().reshape(9, -1), 9, 256, bits)
    np.testing.assert_array_equal(q, np.where(w < 0, -m, m))
    assert q[0, 0] == q[0, 1] == 0 and q[0, 2] > 0 and q[0, 3] < 0


@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("bad", [0.0, float("nan"), float("-inf")])
def test_refused_weights_leave_the_codes(logq, bits, bad):
    W = torch.zeros(16, 256, device="cuda")
    W[7, 9] = bad
    codes = torch.full((logq.logq_packed_bytes(16, 256, bits),), 0x5a, dtype=torch.uint8, device="cuda")
    with pytest.raises(logq.LogqError):
        logq.logq_quantize(W, bits, 2.0, codes=codes)
    assert bool((codes == 0x5a).all())
