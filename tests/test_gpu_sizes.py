"""Component sizes (needs a GPU: -m gpu) at the edges of the counting kernel's units:
words and lanes of a row, batches of eight rows, rows per CTA, counters full to their
last bit, and ties of the largest size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()


@pytest.mark.parametrize("density", [0.0, 0.02, 0.5, 1.0])
@pytest.mark.parametrize("rows,ncols", [(1, 1), (7, 33), (64, 1000), (65, 1024), (1017, 1025), (8129, 70), (3000, 3073), (2049, 4097), (66_000, 5000)])
def test_sizes(rows, ncols, density):
    g = torch.Generator(device="cuda").manual_seed(rows + ncols)
    W = tn.tn_row_words(ncols)
    bits = torch.zeros((rows, W * 64), dtype=torch.bool, device="cuda")
    bits[:, :ncols] = torch.rand((rows, ncols), generator=g, device="cuda") < density
    weights = (1 << torch.arange(8, device="cuda", dtype=torch.int32)).to(torch.uint8)
    S = (bits.view(rows, W * 8, 8).to(torch.uint8) * weights).sum(2, dtype=torch.uint8).view(torch.int64)
    out, ins, best = tn.tn_out_sizes(S, rows, ncols, in_sizes=True, argmax=True)
    want = bits[:, :ncols].sum(0, dtype=torch.int32)
    assert torch.equal(out, want) and torch.equal(ins, bits.sum(1, dtype=torch.int32))
    assert int(best) == int(np.argmax(want.cpu().numpy()))
    assert torch.equal(tn.tn_out_sizes(S, rows, ncols)[0], want)
