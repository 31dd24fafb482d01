"""The GEMM on 256 x 256 tiles of CTA pairs (products of more than one wave of 128 x 128 tiles): edges of its tiles, both layouts of each operand, K
tails and splits, and more tiles than pairs, against numpy and against the 128 x 128 kernel."""
import numpy as np
import pytest

from tests import _parity as P
from tests.test_gpu_warmnet import _bf16_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


@pytest.mark.parametrize("a_km", [True, False])
@pytest.mark.parametrize("b_km", [True, False])
@pytest.mark.parametrize("M,N,K,splits", [
    (2056, 1288, 64, 1),   # one slice; a last tile of 8 rows (the odd CTA has none), 8 columns
    (2184, 1160, 200, 1),  # 8 rows and columns in the odd CTA; a K tail inside a slice
    (1032, 776, 1000, 3),  # uneven K splits
])
def test_pair_gemm_matches_numpy(M, N, K, a_km, b_km, splits):
    import torch
    from paper_1511_04552_gb300.warmstart import gemm_bf16
    r = np.random.default_rng(M + N + K)
    ta, a64 = _bf16_pair(r.normal(size=(M, K) if a_km else (K, M)))
    tb, b64 = _bf16_pair(r.normal(size=(N, K) if b_km else (K, N)))
    A, Bm = a64 if a_km else a64.T, b64 if b_km else b64.T
    kps = ((K + splits - 1) // splits + 63) // 64 * 64
    d = gemm_bf16(ta.cuda(), tb.cuda(), a_km, b_km, splits=splits, k_per_split=kps)
    d = d.cpu().numpy().astype(np.float64)
    for z in range(splits):
        a, b = A[:, z * kps:(z + 1) * kps], Bm[:, z * kps:(z + 1) * kps]
        # FP32 accumulation of exact products: 1e-4 of sum |a||b| as for the other GEMMs
        assert np.all(np.abs(d[z] - a @ b.T) <= 1e-4 * (np.abs(a) @ np.abs(b).T) + 1e-30), z


def test_pair_gemm_many_tiles_equals_small_tiles():
    """160 tiles on at most 76 pairs: a pair goes through its ring and both accumulators several
    times. The 128-column slices of the same product run on 128 x 128 tiles and accumulate in the
    same order: the results are the same bits."""
    import torch
    from paper_1511_04552_gb300.warmstart import gemm_bf16
    g = torch.Generator(device="cuda").manual_seed(1)
    M, N, K = 4096, 2504, 584
    a = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    b = torch.randn(N, K, device="cuda", generator=g).bfloat16()
    d = gemm_bf16(a, b)[0]
    for n0 in range(0, N, 128):
        part = gemm_bf16(a, b[n0:n0 + 128].contiguous())[0]
        assert torch.equal(d[:, n0:n0 + 128], part)
