"""Kernels at the sizes where a tile, a split or a dispatch rule ends, against plain NumPy."""
import numpy as np
import pytest

import paper_2412_14104_gb300 as tg

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    return t


def _dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (12, 12, 12), (16, 16, 16), (17, 15, 33), (36, 36, 1296), (33, 31, 255), (32, 64, 256),
    (65, 3, 257), (3, 65, 273), (432, 72, 36), (1000, 1, 513), (1, 70001, 5), (129, 127, 4099)])
def test_fp64_contraction_tiles_and_splits(torch, M, N, K):
    """Each tile size of the FP64 kernel, ragged edges, the table of K offsets (256 entries)
    and its refills, split K; a transposed A, C accumulated into.  Any order of summation
    stays within (K + 2) eps of sum |a| |b| + |c| (Higham, Accuracy and Stability, Sec. 3.1)."""
    rng = np.random.default_rng(M + 7 * N + 31 * K)
    A, B, C0 = rng.standard_normal((K, M)), rng.standard_normal((K, N)), rng.standard_normal((M, N))
    C = _dev(torch, C0)
    tg.contract([(M, 1, N)], [(N, 1, 1)], [(K, M, N)], _dev(torch, A), _dev(torch, B), C, alpha=0.5, beta=2.0)
    want = 0.5 * (A.T.astype(np.longdouble) @ B.astype(np.longdouble)) + 2.0 * C0
    bound = (K + 4) * EPS * (0.5 * np.abs(A).T @ np.abs(B) + 2.0 * np.abs(C0))
    assert np.all(np.abs(C.cpu().numpy() - want) <= bound)


@pytest.mark.parametrize("K,L", [(16, 16), (17, 31), (5, 103)])
def test_fp64_contraction_permuted_modes(torch, K, L):
    """Two-mode rows, columns and sums with permuted strides, the sum crossing the offset table."""
    I, J, a, b = 5, 7, 3, 4
    rng = np.random.default_rng(K * L)
    A, B = rng.standard_normal((K, I, L, a)), rng.standard_normal((b, L, J, K))
    C = torch.zeros((a, I, b, J), dtype=torch.float64, device="cuda")
    tg.contract([(I, L * a, b * J), (a, 1, I * b * J)], [(J, K, 1), (b, L * J * K, J)],
                [(K, I * L * a, 1), (L, a, J * K)], _dev(torch, A), _dev(torch, B), C)
    want = np.einsum("kila,bljk->aibj", A, B)
    bound = (K * L + 4) * 2 * EPS * np.einsum("kila,bljk->aibj", np.abs(A), np.abs(B))
    assert np.all(np.abs(C.cpu().numpy() - want) <= bound)
