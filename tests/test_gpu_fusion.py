"""Fusion for many sources (needs a GPU: -m gpu) at the edges of its chunks (1,024 and
4,096 sources), of its groups of 256 sources, 32 proxy rows and 256 nodes, for 1 to 64
replicas, and for proxies whose rows do not fit shared memory.  Random proxy matrices,
bit for bit against the oracle's intersection of preimages."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    oracle.build_oracle()


@pytest.mark.parametrize("n,k,R,nsrc", [
    (700, 1, 1, 256), (700, 31, 3, 257), (511, 33, 64, 511), (4000, 1000, 2, 1023), (4000, 1000, 2, 1024), (4000, 65, 5, 1025),
    (5000, 300, 4, 3072), (5000, 300, 4, 3073), (9000, 129, 3, 4096), (9000, 129, 3, 4097), (9000, 2050, 2, 0), (1500, 51_264, 1, 300),
])
def test_estimates(n, k, R, nsrc):
    rng = np.random.default_rng(n + k + nsrc)
    words = tn.tn_row_words(k)
    P = np.zeros((R, k, words), np.uint64)
    full = (k + 63) // 64
    P[:, :, :full] = rng.integers(0, 1 << 63, (R, k, full), dtype=np.uint64) | rng.integers(0, 1 << 63, (R, k, full), dtype=np.uint64) << np.uint64(1)
    if k % 64:
        P[:, :, full - 1] &= np.uint64((1 << (k % 64)) - 1)
    H = rng.integers(0, k, (R, n)).astype(np.uint32)
    src = rng.integers(0, n, nsrc).astype(np.uint32) if nsrc else None
    dP, dH = torch.from_numpy(P.view(np.int64)).cuda(), torch.from_numpy(H.view(np.int32)).cuda()
    est = tn.tn_hash_estimate(dP, R, k, dH, n, src=None if src is None else torch.from_numpy(src.view(np.int32)).cuda())
    ref = oracle.hash_estimate(P[:, :, :full], H, n, src)
    assert np.array_equal(est.cpu().numpy().view(np.uint32), ref)


@pytest.mark.parametrize("max_value", [1, 1022, 1023, 1024, 5000, 2_097_151, 2_097_152, 5_000_000])
def test_error_scan(max_value):
    """Histogram scans of one tile, of several CTAs, and of several tiles per CTA."""
    rng = np.random.default_rng(max_value)
    exact = rng.integers(1, max_value + 1, 4001).astype(np.uint32)
    est = rng.integers(0, max_value + 1, 4001).astype(np.uint32)
    got = tn.tn_error_stats(torch.from_numpy(est.view(np.int32)).cuda(), torch.from_numpy(exact.view(np.int32)).cuda(), max_value)
    assert got["w1_num"] == int(np.abs(np.sort(est).astype(np.int64) - np.sort(exact).astype(np.int64)).sum())
    assert got["sum_abs"] == int(np.abs(est.astype(np.int64) - exact.astype(np.int64)).sum())
