"""Kernels at the sizes where their work splits change: edges of tiles and
lists, remainders, the smallest and the largest of their ranges, against the
oracle (same bars as the other parity tests)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# head statistics: head blocks of 4, 7 and 8 with and without padded heads, one
# pair of blocks to several passes over them, 8 / 16 / 32 tokens a block, rows of
# A on 16 bytes and not, one query, queries that end inside a stage
@pytest.mark.parametrize("H,Hkv,T,gh,gw,B", [
    (1, 1, [1], 5, 7, 1), (3, 1, [33], 6, 6, 1), (5, 5, [9], 9, 9, 1), (28, 4, [31], 7, 9, 1),
    (32, 8, [65], 6, 10, 1), (56, 8, [17], 8, 8, 1), (9, 3, [5, 40], 33, 75, 2),
    (14, 2, [3, 12, 8, 1], 60, 44, 4)])
def test_head_statistics_sizes(H, Hkv, T, gh, gw, B):
    from paper_2608_02134_gb300 import workloads
    from tests.test_gpu_clients import _compare
    wl = workloads.make("qwen", B=B, T=T, gh=gh, gw=gw, D=64, d=32, H=H, Hkv=Hkv, K=9)
    _compare(wl, range(B))


def _clients(kind, B, M, N, seed):
    r = np.random.default_rng(seed)
    if kind == "equal":      # every token its own row of one value: all gains tie in every round
        C = np.zeros((B, M, N), np.float32)
        C[:, np.arange(N) % M, np.arange(N)] = 0.01
        return C
    if kind == "close":      # the same with gains a few units in the last place apart
        C = np.zeros((B, M, N), np.float32)
        v = np.float32(0.01) * (1 + r.permutation(N).astype(np.float32) * np.float32(2.0 ** -22))
        C[:, np.arange(N) % M, np.arange(N)] = v
        return C
    from tests.test_gpu_stages import _structured_clients
    if kind == "dense":      # many survivors a round: lists that start in global memory
        C = r.exponential(size=(B, M, N)) ** 0.25
        return (C / C.sum(axis=(1, 2), keepdims=True)).astype(np.float32)
    return _structured_clients(B, M, N, seed)


# the cluster solver: more equal or nearly equal gains than a round lists exactly
# (the radix search and its ties), lists in global memory, token counts that are no
# multiple of 32, the widest pool, pools that are no power of two, one to sixteen
# CTAs an image, a budget of one round, rounds left over by a fill
@pytest.mark.parametrize("kind,B,M,N,K,b,mult", [
    ("equal", 1, 1200, 1200, 100, 16, 4), ("close", 1, 1300, 1300, 90, 16, 4),
    ("dense", 4, 3000, 1100, 96, 16, 4), ("plain", 1, 500, 33, 20, 16, 4),
    ("plain", 1, 90, 1025, 300, 32, 4), ("plain", 2, 700, 500, 100, 3, 5),
    ("plain", 20, 300, 300, 60, 16, 4), ("plain", 90, 120, 200, 40, 16, 4),
    ("plain", 1, 400, 640, 16, 16, 4), ("plain", 1, 60, 7000, 200, 16, 4),
    ("equal", 1, 40, 700, 64, 16, 4)])
def test_cluster_solver_sizes(kind, B, M, N, K, b, mult):
    from tests.test_gpu_stages import _check_select
    _check_select(_clients(kind, B, M, N, 5 + N), K, batch_b=b, pool_mult=mult)
