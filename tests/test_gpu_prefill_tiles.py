"""The prefill kernel's token tiles (64, 128, 192 or 256 wide), its code copies at
ragged rows, and launches that start before the one they read from has left."""
import pytest
import torch

from paper_2607_01127_gb300 import workloads

from gpu_common import check_linear, lib
from test_gpu_linear import make_layer, reference

pytestmark = pytest.mark.gpu

BASE = {3: 1.25, 4: 1.5, 8: 1.05}


@pytest.fixture(scope="module")
def logq():
    return lib()


# rows on both sides of a lane pair's 16 and a quarter's 32; the last K is a few stages
@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("N,K", [(1, 128), (15, 384), (47, 128), (145, 2048), (300, 640)])
def test_outputs_do_not_depend_on_the_tile_width(logq, bits, N, K):
    """A token's sums run over k in the same order whatever its tile, so batches on
    both sides of each width equal the first rows of a larger one, bit for bit (the
    base workspace leaves k ranges whole)."""
    codes, cb, ocb, q = make_layer(logq, N, K, bits, BASE[bits], N + K)
    X = workloads.activations_torch(600, K, 3, torch.bfloat16, "cuda")
    ws = logq.new_workspace()
    full = logq.logq_linear(codes, cb, X, N, K, workspace=ws)
    Yr, A = reference(X, q, ocb)
    check_linear(full.double().cpu().numpy(), Yr, A, "f32")
    for B in (33, 64, 65, 128, 129, 192, 193, 256, 257, 384, 385, 513, 577):
        assert torch.equal(logq.logq_linear(codes, cb, X[:B].contiguous(), N, K, workspace=ws), full[:B]), B
    assert logq.logq_workspace_status(ws)[0] == logq.LOGQ_OK


@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("B", [40, 200, 700])
def test_chained_launches_wait_for_what_they_read(logq, bits, B):
    """Prefill launches (split k ranges or not) and decode launches of one chain, each
    reading the output before it: without synchronisation, captured and replayed, the
    same bits as with the stream drained after every call."""
    n = 1024
    codes, cb, _, _ = make_layer(logq, n, n, bits, BASE[bits], 8)
    x0 = workloads.activations_torch(B, n, 9, torch.bfloat16, "cuda")
    wide = logq.new_workspace(None, logq.logq_linear_workspace_bytes(B, n, n, bits))
    base = logq.new_workspace()
    bufs = [torch.empty(B, n, dtype=torch.bfloat16, device="cuda") for _ in range(12)]

    def chain(sync):
        x = x0
        for i, y in enumerate(bufs):
            if i % 3 == 2:          # a few rows through the decode kernel, the rest copied
                y.copy_(x)
                logq.logq_linear(codes, cb, x[:16], n, n, y_dtype=torch.bfloat16, Y=y[:16], workspace=base)
            else:
                logq.logq_linear(codes, cb, x, n, n, y_dtype=torch.bfloat16, Y=y, workspace=(wide, base)[i % 2])
            if sync:
                torch.cuda.synchronize()
            x = y

    chain(True)
    want = [y.clone() for y in bufs]
    chain(False)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(bufs, want))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(False)
    for y in bufs:
        y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(bufs, want))
