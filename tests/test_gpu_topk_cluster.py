"""dkv_topk_mask around the sizes where its kernels change over: one cluster of 8
CTAs x 1024 threads with 8, 16 or 32 keys a thread, then the grid-wide kernel. Bit
for bit against the oracle's global Top-K, as everywhere."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_32663_gb300.dkv as dkv

pytestmark = pytest.mark.gpu
THREADS = 8 * 1024


@pytest.fixture(scope="module", autouse=True)
def _built(cuda):
    from paper_2609_32663_gb300 import build
    build.build_library()
    torch.cuda.set_device(cuda)


def values(kind, n):
    rng = np.random.default_rng([n, len(kind)])
    if kind == "probabilities":
        return (1 / (1 + np.exp(-2 * rng.standard_normal(n)))).astype(np.float32)
    if kind == "any bits":  # every exponent, both signs, infinities, NaN
        return rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32).view(np.float32)
    return rng.choice(np.array([0.0, -0.0, np.nan, np.inf, -np.inf, 0.5, 0.25], np.float32), n)


@pytest.mark.parametrize("kind", ["probabilities", "any bits", "ties"])
@pytest.mark.parametrize("n", [1, 7, 127, 129, 513, THREADS - 1, THREADS + 1, 8 * THREADS - 1, 8 * THREADS,
                               8 * THREADS + 1, 16 * THREADS, 16 * THREADS + 1, 32 * THREADS, 32 * THREADS + 1])
def test_sizes_at_the_kernels_edges(n, kind, cuda):
    P = values(kind, n)
    Pd = torch.from_numpy(P).to(cuda)
    for K in sorted({1, n // 3, n - 1} - {0, n}):
        M = torch.full((n + 16,), 7, dtype=torch.uint8, device=cuda)  # the bytes past n stay
        ws = torch.full((dkv.dkv_topk_workspace_bytes() // 4,), -1, dtype=torch.int32, device=cuda)
        dkv.dkv_topk_mask(Pd, K, M[:n], ws)
        got = M.cpu().numpy()
        assert np.array_equal(got[:n], O.topk_mask(P, K)) and (got[n:] == 7).all(), (n, K)
        assert int(ws[0].item()) == 0


def test_unaligned_views_and_replay_in_a_graph(cuda):
    n = 70001
    P = values("probabilities", n + 3)
    Pd = torch.from_numpy(P).to(cuda)[3:]
    M = torch.zeros(n + 1, dtype=torch.uint8, device=cuda)[1:]
    ws = torch.zeros(dkv.dkv_topk_workspace_bytes() // 4, dtype=torch.int32, device=cuda)
    dkv.dkv_topk_mask(Pd, 1000, M, ws)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dkv.dkv_topk_mask(Pd, n // 2, M, ws)
    for seed in (1, 2):
        fresh = np.random.default_rng(seed).random(n).astype(np.float32)
        Pd.copy_(torch.from_numpy(fresh))
        graph.replay()
        assert np.array_equal(M.cpu().numpy(), O.topk_mask(fresh, n // 2))
