"""The decode kernel at the edges of its launch shapes: against the oracle, with a
bound on its fp32 sums.

Bound: a product is exact; an output is a sum of K of them.  Each 16-term
tensor-core sum truncates its terms at 2^-23 of the largest and its result, chains
of at most 2 follow, then at most 4 + 3 pairwise additions, one per span of a warp
(at most 14336 / 1024 / 8 + 1) and 8 + 8 over partial sums and parts, each rounding
at 2^-24 of its operands: below 60 * 2^-24 of sum_k |x_k w_k|."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_01127_gb300 import workloads

from gpu_common import lib
from test_gpu_linear import make_layer, reference

pytestmark = pytest.mark.gpu

BOUND = 60 * 2.0 ** -24
BASE = {3: 1.25, 4: 1.5, 8: 1.05}


@pytest.fixture(scope="module")
def logq():
    return lib()


def check(Y, Yr, A):
    err = np.abs(Y.double().cpu().numpy() - Yr)
    assert np.all(err <= BOUND * A), float((err / A).max())


# batches on both sides of each padded size; rows around a tile and a CTA's share;
# K below, at and above a span of each shape
@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("N,K", [(1, 128), (17, 384), (305, 3968), (304, 4096), (129, 14336), (5000, 640)])
def test_decode_shapes(logq, bits, B, N, K):
    codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], N + K + B)
    X = workloads.activations_torch(B, K, B, torch.float16 if (B + N) % 2 else torch.bfloat16, "cuda")
    check(logq.logq_linear(codes, cb, X, N, K), *reference(X, q, ocb))


@pytest.mark.parametrize("bits,B,N,K", [(4, 17, 1024, 4096), (3, 32, 2048, 2048), (8, 24, 1024, 4096), (4, 1, 2114, 3968), (4, 1, 65536, 128),
                                           (3, 1, 2114, 3968), (4, 2, 1024, 4096), (8, 1, 32768, 128)])
def test_both_sides_of_a_dispatch_line(logq, bits, B, N, K):
    """N rows are the most of the one path (batches above 16: up to 4 M weights; one CTA
    per SM: up to 4 M; short rows at batch 1, 3 and 4 bits: up to 8 M); one more row takes
    the other."""
    codes, cb, ocb, q = make_layer(logq, N + 1, K, bits, BASE[bits], 1)
    X = workloads.activations_torch(B, K, 2, torch.bfloat16, "cuda")
    more = logq.logq_linear(codes, cb, X, N + 1, K)
    fewer = logq.logq_linear(codes[:logq.logq_packed_bytes(N, K, bits)].clone(), cb, X, N, K)
    rows = np.r_[0:64, N - 64:N]
    Yr, A = reference(X, q[rows], ocb)
    check(fewer[:, rows], Yr, A)
    if B <= 16:
        check(more[:, rows], Yr, A)
    else:          # the tensor-memory kernel's chains truncate K / 16 times
        assert np.all(np.abs(more[:, rows].double().cpu().numpy() - Yr) <= (K / 16 + 60) * 2.0 ** -23 * A)


# few rows of long K (the rows that each CTA takes one by one) and one more than the most of
# them at each width; k of whole spans, of a ragged last one and on both sides of the line
@pytest.mark.parametrize("bits,B", [(4, 3), (4, 4), (4, 5), (4, 8), (4, 9), (4, 16), (3, 3), (3, 4), (8, 3), (8, 4)])
@pytest.mark.parametrize("N,K", [(1, 14336), (2, 2048), (3, 2176), (128, 4224), (129, 3968), (256, 4096), (257, 4096), (384, 8576),
                                 (385, 8576)])
def test_few_rows(logq, bits, B, N, K):
    codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], N + K)
    X = workloads.activations_torch(B, K, B, torch.float16 if B % 2 else torch.bfloat16, "cuda")
    Y = logq.logq_linear(codes, cb, X, N, K)
    check(Y, *reference(X, q, ocb))
    # grouped: the same rows as three matrices
    if N == 128:
        row = logq.logq_packed_bytes(1, K, bits)
        parts = [(codes[a * row:b * row].clone(), cb, b - a, None) for a, b in ((0, 1), (1, 100), (100, 128))]
        assert torch.equal(torch.cat(logq.logq_linear_grouped(parts, X, K), 1), Y)


@pytest.mark.parametrize("bits", [3, 4, 8])
def test_infinite_levels_stay_out_of_the_ragged_end(logq, bits):
    """fp16 levels that overflow: outputs over a last span that K leaves ragged are those
    of the infinities in the matrix, not NaN from lanes past K."""
    N, K = 5, 4224
    cb = logq.logq_build_codebook(bits, 1.3, 1e6)
    codes = torch.zeros(logq.logq_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
    codes.view(N, -1)[:, 0] = cb.qmax                       # k = 0: the largest level, +inf in fp16
    for B in (4, 16):
        X = torch.ones(B, K, dtype=torch.float16, device="cuda")
        assert bool((logq.logq_linear(codes, cb, X, N, K) == float("inf")).all())


# k on both sides of the lines between the shapes for short rows; fewer rows than a CTA's
# warps have tiles for, and more
@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("B", [1, 2, 4])
@pytest.mark.parametrize("K", [1024, 1152, 2048, 2176, 4096, 4224])
def test_short_rows(logq, bits, B, K):
    for N in (3, 2000):
        codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], K + B)
        X = workloads.activations_torch(B, K, B, torch.bfloat16, "cuda")
        check(logq.logq_linear(codes, cb, X, N, K), *reference(X, q, ocb))


@pytest.mark.parametrize("bits,B,N,K", [(4, 3, 21001, 2048), (4, 4, 33000, 2048), (8, 4, 47001, 1024), (4, 16, 60011, 128)])
def test_rows_of_a_cta_in_chunks(logq, bits, B, N, K):
    """More rows per CTA than its partial sums have room for: equal chunks, ragged ends."""
    codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], 9)
    X = workloads.activations_torch(B, K, 3, torch.bfloat16, "cuda")
    Y = logq.logq_linear(codes, cb, X, N, K)
    rows = np.r_[0:400, N // 2:N // 2 + 300, N - 300:N]
    Yr, A = reference(X, q[rows], ocb)
    check(Y[:, rows], Yr, A)
    part = logq.logq_linear(codes[:logq.logq_packed_bytes(999, K, bits)].clone(), cb, X, 999, K)
    assert torch.equal(Y[:, :999], part)             # a row's sums do not depend on the chunks


@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("B", [9, 16, 32])
@pytest.mark.parametrize("sets", [0, 1, 2, 3, 8])
def test_parts_of_k_use_the_workspace_given(logq, bits, B, sets):
    """Room for `sets` partial sums of every output, less 4 bytes for one of them;
    nothing past the stated size is written."""
    N, K = 203, 14336
    codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], 4)
    X = workloads.activations_torch(B, K, 5, torch.bfloat16, "cuda")
    nbytes = logq.logq_workspace_bytes() + sets * 4 * B * N - (4 if sets == 2 else 0)
    room = torch.full((nbytes + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    room[:logq.logq_workspace_bytes()] = 0
    Y = logq.logq_linear(codes, cb, X, N, K, workspace=room[:nbytes])
    check(Y, *reference(X, q, ocb))
    assert bool((room[nbytes:] == 0x5a).all())
    st, _ = logq.logq_workspace_status(room[:nbytes])
    assert st == logq.LOGQ_OK


@pytest.mark.parametrize("K", [1152, 4224])
@pytest.mark.parametrize("B", [1, 2, 4, 8, 16, 32])
def test_non_finite_activations_stay_in_their_row(logq, B, K):
    """A NaN or an infinity reaches every output of its own batch row (an infinity as
    NaN where the level is 0) and no other row, although rows and parts of K share
    one matrix instruction."""
    N = 70
    codes, cb, ocb, q = make_layer(logq, N, K, 4, 1.5, 6)
    X = workloads.activations_torch(B, K, 7, torch.bfloat16, "cuda")
    clean = logq.logq_linear(codes, cb, X, N, K)
    for b in range(0, B, 3):
        for k, v in ((0, float("nan")), (K - 1, float("inf"))):
            Xb = X.clone()
            Xb[b, k] = v
            Y = logq.logq_linear(codes, cb, Xb, N, K)
            keep = [i for i in range(B) if i != b]
            assert torch.equal(Y[keep], clean[keep])
            w = oracle.dequant(q, ocb, oracle.TABLE_BF16)[:, k]
            want = np.full(N, np.nan) if np.isnan(v) else np.where(w == 0, np.nan, np.copysign(np.inf, w))
            np.testing.assert_array_equal(Y[b].double().cpu().numpy(), want)
