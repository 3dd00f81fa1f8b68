"""The GPTQ kernels at the edges of their tiles: the factor over many diagonal blocks,
where the triangular products change tile size, and with pivots of any magnitude; the
quantisation where the column update changes tile size, and at the largest K of use."""
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


def test_factor_of_many_blocks(logq):
    """K = 3328: 52 diagonal blocks, trailing updates of 1326 to 1 tiles of 64 x 64, the
    inverse in 64 x 64 tiles with shortened pairs.  Bound as for the smaller sizes."""
    K = 3328
    Hf = hessian(K, 11, T=K + 64).astype(np.float32)
    U, _ = logq.gptq_factor(torch.from_numpy(Hf).cuda(), 0.01)
    U = U.double().cpu().numpy()
    Uo = oracle.gptq_factor(Hf.astype(np.float64), 0.01)
    assert np.all(np.tril(U, -1) == 0.0)
    assert float(np.max(np.abs(U - Uo)) / np.max(np.abs(Uo))) < 2e-4


def device_hessian(K, T, seed):
    """hessian() made on the device, in fp64: T inputs."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(T, K, device="cuda", generator=g, dtype=torch.float64)
    X *= 1.0 + torch.rand(K, device="cuda", generator=g, dtype=torch.float64)
    X[:, 1:] += 0.5 * X[:, :-1].clone()
    return X.T @ X


@pytest.mark.parametrize("K", [6016, 8192])
def test_factor_in_the_large_tiles(logq, K):
    """The last levels of the triangular inverse take 64 x 128 tiles from two 128 x 128
    tiles per SM on: at 8192 a whole pair (4096 rows a side), at 6016 a shortened one
    (4096 and 1920).  Hd^-1 = U^T U: against the same steps in fp64, and U Hd U^T = I on
    random vectors.  Bounds as for the smaller sizes."""
    Hf = device_hessian(K, K + 64, K).float()
    U, dead = logq.gptq_factor(Hf, 0.01)
    assert not bool(dead.any()) and bool((torch.tril(U, -1) == 0).all())
    Hd = Hf.double()
    Hd.diagonal().add_(0.01 * Hd.diagonal().mean())
    # J Hd J = L L^T (J reverses), U = J L^-1 J
    L = torch.linalg.cholesky(Hd.flip(0, 1))
    want = torch.linalg.solve_triangular(L, torch.eye(K, device="cuda", dtype=torch.float64), upper=False).flip(0, 1)
    assert float((U.double() - want).abs().max() / want.abs().max()) < 2e-4
    v = torch.randn(K, 8, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(1))
    got = U.double() @ (Hd @ (U.double().T @ v))
    assert float((got - v).norm() / v.norm()) < 2e-4


def test_gptq_of_a_wide_matrix(logq):
    """K = 14336 (an MLP's output projection): factor and quantisation; the factor against
    64 bits on random vectors, the first rows' codes against the oracle's column loop on
    the device's factor."""
    K, N = 14336, 600
    Hf = device_hessian(K, K + 256, 5).float()
    W = torch.from_numpy(workloads.weights_np(N, K, seed=12, outliers=True)).cuda()
    cb = logq.logq_build_codebook(4, 1.6, float(W.abs().max()))
    U, _ = logq.gptq_factor(Hf, 0.01)
    Hd = Hf.double()
    Hd.diagonal().add_(0.01 * Hd.diagonal().mean())
    v = torch.randn(K, 4, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(2))
    got = U.double() @ (Hd @ (U.double().T @ v))
    assert float((got - v).norm() / v.norm()) < 2e-4
    codes = logq.logq_gptq(W, Hf, cb).cpu().numpy().reshape(N, -1)
    q = oracle.unpack(codes, N, K, 4)
    rows = [0, 1, 299, N - 1]
    # the same column loop in fp64 (numpy), blocks of 256 columns
    Ud = U.double().cpu().numpy()
    tau = np.array(cb.thresh[:cb.qmax], np.float32).astype(np.float64)
    level = np.array(cb.level[:8], np.float32).astype(np.float64)
    w = W.cpu().numpy()[rows].astype(np.float64)
    want = np.zeros((len(rows), K), int)
    for j0 in range(0, K, 256):
        E = np.zeros((len(rows), 256))
        for j in range(j0, j0 + 256):
            m = (np.abs(w[:, j, None]) >= tau).sum(1)
            want[:, j] = np.where(w[:, j] < 0, -m, m)
            E[:, j - j0] = (w[:, j] - np.where(w[:, j] < 0, -level[m], level[m])) / Ud[j, j]
            w[:, j + 1:j0 + 256] -= E[:, j - j0, None] * Ud[j, j + 1:j0 + 256]
        w[:, j0 + 256:] -= E @ Ud[j0:j0 + 256, j0 + 256:]
    # fp32 and fp64 put a few weights on different sides of a boundary, and the rest of the
    # row follows: the agreement that test_gptq_matches_oracle asks for
    assert float(np.mean(q[rows] == want)) >= 0.98


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
