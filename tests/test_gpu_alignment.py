"""Inputs at the alignment of their own type (needs a GPU: -m gpu): calls that read
matrices and sketches in 16-byte loads also take a buffer that starts anywhere a value
may start, with the same results."""
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


def shifted(x, by):
    """A copy of x that starts `by` elements behind a 16-byte boundary."""
    room = torch.zeros(x.numel() + 16, dtype=x.dtype, device="cuda")
    assert room.data_ptr() % 16 == 0
    y = room[by : by + x.numel()].view(x.shape)
    y.copy_(x)
    assert y.data_ptr() % 16 == by * x.element_size() % 16
    return y


@pytest.mark.parametrize("n,k,R,nsrc", [(700, 33, 3, 40), (700, 33, 3, 257), (1100, 300, 2, 1025), (9000, 129, 3, 4097)])
def test_proxies(n, k, R, nsrc):
    rng = np.random.default_rng(n + k)
    full = (k + 63) // 64
    P = np.zeros((R, k, tn.tn_row_words(k)), np.uint64)
    P[:, :, :full] = rng.integers(0, 1 << 63, (R, k, full), dtype=np.uint64)
    P[:, :, full - 1] &= np.uint64((1 << (k % 64 or 64)) - 1)
    H = rng.integers(0, k, (R, n)).astype(np.uint32)
    src = rng.integers(0, n, nsrc).astype(np.uint32)
    dP, dH = shifted(torch.from_numpy(P.view(np.int64)), 1), torch.from_numpy(H.view(np.int32)).cuda()
    est = tn.tn_hash_estimate(dP, R, k, dH, n, src=torch.from_numpy(src.view(np.int32)).cuda())
    assert np.array_equal(est.cpu().numpy().view(np.uint32), oracle.hash_estimate(P[:, :, :full], H, n, src))


@pytest.mark.parametrize("p", [4, 5, 10])
@pytest.mark.parametrize("by", [1, 8])
def test_sketches(p, by):
    n = 300
    rng = np.random.default_rng(p)
    R = torch.from_numpy(rng.integers(0, 62 - p, (n, 8 * tn.tn_row_words(8 << p))).astype(np.uint8))
    aligned = tn.tn_hll_estimate(R.cuda(), n, p)
    assert torch.equal(tn.tn_hll_estimate(shifted(R, by), n, p), aligned)  # the sum is exact in both


@pytest.mark.parametrize("rows,ncols", [(65, 1000), (300, 3073), (8200, 4096)])
def test_sizes(rows, ncols):
    rng = np.random.default_rng(ncols)
    W = tn.tn_row_words(ncols)
    bits = np.zeros((rows, 64 * W), np.uint8)
    bits[:, :ncols] = rng.random((rows, ncols)) < 0.3
    S = torch.from_numpy(np.packbits(bits, axis=1, bitorder="little").view(np.int64))
    out, ins, best = tn.tn_out_sizes(shifted(S, 1), rows, ncols, in_sizes=True, argmax=True)
    want = bits.sum(0)[:ncols]
    assert np.array_equal(out.cpu().numpy(), want) and np.array_equal(ins.cpu().numpy(), bits.sum(1))
    assert int(best) == int(np.argmax(want))
