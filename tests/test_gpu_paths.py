"""The branches of the kernels' dispatch at the sizes where they can go wrong,
through the C ABI, against plain products and the oracle's definitions."""
import numpy as np
import pytest

import workloads as wl
from oracle import tadm_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2609_37924_gb300 import tadm
    return tadm


def bf16_tensor(shape, seed, std=1.0):
    bits = wl.normal(seed, 99, int(np.prod(shape)), 0.0, std, "bf16").reshape(shape)
    return torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda(), O.widen(bits)


# fp32 outputs leave through TMA stores of 32 x 32 boxes (N % 4 == 0 and
# ldc % 4 == 0: TMA clips to 16 bytes, not to elements), otherwise row by row:
# ragged edges, padding columns that must stay untouched, an odd stride
@pytest.mark.parametrize("M,N,K,ldc", [(33, 300, 72, 304), (33, 301, 72, 304), (33, 301, 72, 301),
                                       (257, 260, 136, 260), (130, 36, 64, 40), (1, 4, 8, 4), (1, 1, 8, 4)])
def test_gemm_fp32_store_edges(T, M, N, K, ldc):
    A, a = bf16_tensor((M, K), 1)
    B, b = bf16_tensor((N, K), 2)
    flat = torch.full((M * ldc + 8,), 7.0, dtype=torch.float32, device="cuda")
    C = flat[:M * ldc].view(M, ldc)
    T.tadm_gemm(A, B, C[:, :N], dtype=1)
    got = C.cpu().numpy().astype(np.float64)
    # fp32 accumulation of K exact bf16 products
    assert np.abs(got[:, :N] - a @ b.T).max() <= 1e-5 * np.abs(a).max() * np.abs(b).max() * np.sqrt(K)
    assert (got[:, N:] == 7.0).all() and (flat[M * ldc:] == 7.0).all().item()
