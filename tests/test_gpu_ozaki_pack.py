"""The packing of the FP64-accurate product around its steps: one pass up to K = 128,
two above it, the last step short, one row block and several, zero rows and columns,
a workspace beyond the pool's, and calls from several threads on their own streams."""
import threading

import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from parity_util import have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def integers(M, N, K, seed):
    """Products of 11-bit integers: every sum is exact, here and in FP64."""
    import torch
    rng = np.random.default_rng(seed)
    A = rng.integers(-1024, 1025, size=(M, K)).astype(np.float64)
    B = rng.integers(-1024, 1025, size=(K, N)).astype(np.float64)
    A[M // 2] = 0.0
    B[:, N // 3] = 0.0
    return A, B, torch.from_numpy(np.ascontiguousarray(A.T)).cuda(), torch.from_numpy(np.ascontiguousarray(B.T)).cuda()


def product(M, N, K, dA, dB, stream=None):
    import torch
    C = torch.full((N, M), 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    eng.cmaes_ozaki_dgemm(M, N, K, 1.0, dA.data_ptr(), M, dB.data_ptr(), K, 0.0, C.data_ptr(), M, stream)
    return C.T.cpu().numpy()


@pytest.mark.parametrize("K", [1, 31, 32, 127, 128, 129, 160, 255, 257, 2049])
@pytest.mark.parametrize("M,N", [(1, 1), (63, 65), (64, 128), (200, 130)])
def test_steps_of_k(M, N, K):
    A, B, dA, dB = integers(M, N, K, 100 * M + K)
    assert np.array_equal(product(M, N, K, dA, dB), A @ B)


def test_workspace_beyond_the_pool():
    M, N, K = 2048, 64, 3072  # 2048 x 3072 x 14 bytes = 84 MiB
    A, B, dA, dB = integers(M, N, K, 5)
    for _ in range(2):
        assert np.array_equal(product(M, N, K, dA, dB), A @ B)


def test_threads():
    import torch
    jobs = [integers(96 + 32 * t, 70, 200 + 50 * t, t) for t in range(4)]
    bad = []

    def work(t):
        A, B, dA, dB = jobs[t]
        stream = torch.cuda.Stream()
        for _ in range(20):
            if not np.array_equal(product(A.shape[0], B.shape[1], A.shape[1], dA, dB, stream.cuda_stream), A @ B):
                bad.append(t)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
