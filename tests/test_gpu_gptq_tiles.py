"""The GPTQ kernels at the edges of their tiles: the factor where the trailing
updates change tile size and with pivots of any magnitude, the quantisation where
the column update does."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_01127_gb300 import workloads

from gpu_common import lib
from test_gpu_gptq import hessian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def logq():
    return lib()


def test_factor_beyond_the_small_tiles(logq):
    """K = 3328: 128 x 128 tiles for the first trailing updates (26 x 26 / 2 tiles,
    more than two per SM), 64 x 64 for the rest.  Bound as for the smaller sizes."""
    K = 3328
    Hf = hessian(K, 11, T=K + 64).astype(np.float32)
    U, _ = logq.gptq_factor(torch.from_numpy(Hf).cuda(), 0.01)
    U = U.double().cpu().numpy()
    Uo = oracle.gptq_factor(Hf.astype(np.float64), 0.01)
    assert np.all(np.tril(U, -1) == 0.0)
    assert float(np.max(np.abs(U - Uo)) / np.max(np.abs(Uo))) < 2e-4


@pytest.mark.parametrize("power", [-80, 80])
def test_factor_scales_exactly(logq, power):
    """H times 4^s gives U times 2^-s, bit for bit: every step is a product, a sum or
    a quotient of scaled values."""
    Hf = hessian(256, 3).astype(np.float32)
    U, _ = logq.gptq_factor(torch.from_numpy(Hf).cuda(), 0.01)
    S, _ = logq.gptq_factor(torch.from_numpy(Hf * np.float32(2.0 ** power)).cuda(), 0.01)
    assert torch.equal(S, U * 2.0 ** (-power // 2))


@pytest.mark.parametrize("bits", [4, 8])
def test_rows_do_not_depend_on_the_tiles(logq, bits):
    """Rows are quantised independently and a sum's order does not depend on the
    tile, so 4999 rows (64 x 128 tiles, more than two 128 x 128 per SM) equal
    their slices of 17 and 1000 rows (64 x 64)."""
    K, N = 1664, 4999
    H = torch.from_numpy(hessian(K, 5, T=2 * K).astype(np.float32)).cuda()
    W = torch.from_numpy(workloads.weights_np(N, K, seed=9)).cuda()
    cb = logq.logq_build_codebook(bits, {4: 2.0, 8: 1.05}[bits], float(W.abs().max()))
    codes = logq.logq_gptq(W, H, cb).view(N, -1)
    for r0, n in ((0, 1), (0, 17), (3000, 1000), (N - 1000, 1000)):
        part = logq.logq_gptq(W[r0:r0 + n].contiguous(), H, cb).view(n, -1)
        assert torch.equal(part, codes[r0:r0 + n])


@pytest.mark.parametrize("bits,B,N", [(4, 8, 132000), (4, 16, 33000), (4, 17, 9000), (4, 40, 9000), (8, 5, 9000),
                                      (8, 16, 9000), (8, 40, 9000)])
def test_linear_right_after_gptq(logq, bits, B, N):
    """Launches that keep to stream order (4 bits: 8 rows of more than 32 M weights, 16 of
    more than 8 M) read the codes that GPTQ has just written, in the decode kernel and in
    the prefill kernel."""
    K = 256
    H = torch.from_numpy(hessian(K, 6, T=2 * K).astype(np.float32)).cuda()
    W = torch.from_numpy(workloads.weights_np(N, K, seed=10)).cuda()
    cb = logq.logq_build_codebook(bits, {4: 2.0, 8: 1.05}[bits], float(W.abs().max()))
    X = workloads.activations_torch(B, K, 11, torch.bfloat16, "cuda")
    codes = logq.logq_gptq(W, H, cb)
    want = logq.logq_linear(codes, cb, X, N, K)
    ws = logq.new_workspace(None, logq.logq_linear_workspace_bytes(B, N, K, bits))
    for _ in range(10):
        codes.zero_()
        torch.cuda.synchronize()
        logq.logq_gptq(W, H, cb, codes=codes)
        got = logq.logq_linear(codes, cb, X, N, K, workspace=ws)
        assert torch.equal(got, want)
