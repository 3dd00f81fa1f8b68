"""w_min where the counting passes of the energy selection can go wrong: against
the oracle's, exactly (the cumulative share at every data value near the crossing
is far from eps, so there is no near-tie)."""
import numpy as np
import pytest
import torch

from paper_2607_01127_gb300 import workloads

from gpu_common import lib
from test_gpu_energy import check_wmin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def logq():
    return lib()


def stretch(n, high):
    """Most of an exponent's weights at its start and `high` of them, of as many
    energies, in its upper half: the counts leave a window of hundreds of buckets."""
    rng = np.random.default_rng(n + high)
    w = np.concatenate([rng.uniform(1.0, 1.01, n - high), rng.uniform(1.5, 2.0, high)]).astype(np.float32)
    return rng.permutation(w) * np.where(rng.random(n) < 0.5, -1.0, 1.0).astype(np.float32)


def share_below(w, t):
    a = np.abs(w.astype(np.float64)).ravel()
    return float(np.sum(a[a < t] ** 2) / np.sum(a * a))


def scales(n, share, small):
    return np.where(np.random.default_rng(n).random(n) < share, small, 1.0).astype(np.float32)


CASES = {
    # the window does not settle the crossing: exact bucket energies do
    "stretch": lambda: stretch(1024 * 128, 400).reshape(1024, 128),
    "stretch_subnormal": lambda: np.float32(2.0 ** -128) * stretch(64 * 384, 60).reshape(64, 384),
    # every CTA's first values far below, or above, most of the others: outside pass 1's window
    "late_large": lambda: np.concatenate([np.full((600, 4096), 1e-25, np.float32),
                                          workloads.weights_np(300, 4096, seed=3)]),
    "early_large": lambda: np.concatenate([workloads.weights_np(2, 128, seed=4) * np.float32(1e20),
                                           workloads.weights_np(37, 128, seed=5)]),
    # rows or columns of dead neurons: below the windows (where the crossing may lie: 0.2) or windows' first values
    "dead_rows": lambda: workloads.weights_np(900, 1024, seed=8) * scales(900, 0.3, 1e-14)[:, None],
    "dead_rows_subnormal": lambda: workloads.weights_np(900, 1024, seed=8) * scales(900, 0.95, 1e-38)[:, None],
    "dead_columns": lambda: workloads.weights_np(900, 1024, seed=8) * scales(1024, 0.1, 1e-25)[None, :],
    # windows that move up again and again
    "ascending": lambda: workloads.weights_np(1500, 512, seed=9) * np.exp2(np.arange(1500) // 8 - 100.0).astype(np.float32)[:, None],
    # one vector, a grid's remainder, zeros in every vector
    "one_row": lambda: workloads.weights_np(1, 128, seed=6),
    "zeros": lambda: workloads.weights_np(129, 640, seed=7) * (np.arange(640) % 4 == 1).astype(np.float32),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("where", [0.2, 0.999])
def test_energy_wmin_in_hard_distributions(logq, name, where):
    w = CASES[name]()
    a = np.unique(np.abs(w))
    a = a[a > 0]
    t = float(a[min(int(where * len(a)), len(a) - 2)])       # eps half way through this value's energy
    eps = 0.5 * (share_below(w, t) + share_below(w, float(np.nextafter(np.float32(t), np.float32(np.inf)))))
    _, cb, wmin = logq.logq_quantize_energy(torch.from_numpy(np.ascontiguousarray(w)).cuda(), 4, eps)
    assert check_wmin(w, eps, wmin) and wmin == t
    assert cb.range == float(np.abs(w).max())
