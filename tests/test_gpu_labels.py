"""The label kernel's two forms (16-byte rows and others) against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_seq,length,heads,shift", [
    (1, 4, 0, 0), (2, 508, 10, 0), (3, 512, 1, 0), (2, 516, 64, 0), (1, 1024, 3, 0),      # aligned rows: edges of a block's columns, no heads, the most
    (2, 513, 10, 0), (3, 255, 16, 0), (2, 512, 10, 1), (1, 8, 12, 0),                     # lengths and a matrix off the boundary, more heads than tokens
])
def test_labels(n_seq, length, heads, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle.labels import syntax_enriched_labels
    from paper_2503_14153_b200 import binding as B
    rng = np.random.default_rng(n_seq * length + heads)
    tok = rng.integers(8, 100, (n_seq, length)).astype(np.int32)
    tok[rng.random(tok.shape) < 0.2] = 7
    want = np.stack([syntax_enriched_labels(t, heads, 7, 0, -100) for t in tok])
    flat = torch.full((want.size + 8,), -7, dtype=torch.int32, device="cuda")
    t = torch.from_numpy(tok).cuda()
    rc = B.load_library().spec_build_labels(t.data_ptr(), n_seq, length, heads, 7, 0, -100, flat.data_ptr() + 4 * shift, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    got = flat.cpu().numpy()
    assert rc == 0 and (got[:shift] == -7).all() and (got[shift + want.size:] == -7).all()
    assert np.array_equal(got[shift:shift + want.size].reshape(want.shape), want)
