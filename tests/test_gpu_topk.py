"""Candidate lists out of the tiles' maxima, against the heads' logits in 64 bits."""
import numpy as np
import pytest

from synthetic import draw_prompt, draw_weights, get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,batch,kmax", [
    (1160, 1, 10), (1290, 3, 10),             # ten and eleven tiles for ten candidates
    (1000, 1, 10),                            # too few tiles: the slices' kernel
    (8192, 2, 16), (8200, 2, 16),             # the most tiles that are groups of their own, and one more
    (32016, 16, 1), (32017, 5, 3), (37888, 1, 16),
])
def test_candidates(vocab, batch, kmax):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="topk", dtype="bf16", vocab=vocab, d_ffn=704, n_heads=2, n_kv_heads=2, head_dim=128, n_medusa=1, topk=(kmax,), tree_nodes=kmax + 1, seed=6)
    w = draw_weights(cfg)
    dec = SpecDecoder(cfg, upload_weights(cfg, w), build_tree(cfg.topk, kmax + 1), 64, max_batch=batch)
    dec.prefill([draw_prompt(cfg.with_(seed=30 + b), 5 + b) for b in range(batch)])
    h = torch.from_numpy(dec.debug(B.DBG_H_LAST)).bfloat16().double()
    dec.set_option(B.OPT_TRACE, 1)
    dec.step()
    assert (("topk_tiles" if vocab > 1000 else "topk_slices_tc") in [r[0] for r in dec.trace()])
    cand = dec.debug(B.DBG_CAND)
    assert dec.kmax == kmax
    dec.close()

    def operand(a):
        return torch.from_numpy(np.ascontiguousarray(a)).bfloat16().double()
    r = (h + torch.nn.functional.silu(h @ operand(w["medusa.0.w"]).T + operand(w["medusa.0.b"]))).bfloat16().double()
    z = (r @ operand(w["lm_head"]).T).numpy()
    for b in range(batch):
        got = cand[b, 1]
        assert len(set(got.tolist())) == kmax
        # (a rounding of r that falls the other way moves a logit by 2^-9 of one of its 256 products)
        tol = 2.0 ** -8 * np.abs(z[b]).max() / 16
        picked = z[b][got]
        assert (np.diff(picked) <= tol).all()
        assert np.delete(z[b], got).max() <= picked[-1] + tol


@pytest.mark.parametrize("vocab,batch,kmax,classes", [
    (2371, 1, 10, 0), (3001, 2, 5, 0),        # the fewest columns whose warps keep their rows, a ragged end
    (32016, 3, 4, 0), (32016, 9, 16, 0),      # up to four rows, and two groups of eight
    (9001, 1, 10, 7), (9001, 6, 16, 7),       # more equal values than the lists hold
])
def test_candidates_float32(vocab, batch, kmax, classes):
    """The same in float32, whose tiles are every so many-th piece of the vocabulary: equal values go by their index."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="topk", vocab=vocab, d_ffn=704, n_heads=2, n_kv_heads=2, n_medusa=1, topk=(kmax,), tree_nodes=kmax + 1, seed=7)
    w = draw_weights(cfg)
    if classes:
        w["lm_head"] = np.ascontiguousarray(w["lm_head"][np.arange(vocab) % classes])
    dec = SpecDecoder(cfg, upload_weights(cfg, w), build_tree(cfg.topk, kmax + 1), 64, max_batch=batch)
    dec.prefill([draw_prompt(cfg.with_(seed=30 + b), 5 + b) for b in range(batch)])
    h = torch.from_numpy(dec.debug(B.DBG_H_LAST)).double()
    dec.set_option(B.OPT_TRACE, 1)
    dec.step()
    assert "topk_tiles" in [r[0] for r in dec.trace()]
    cand = dec.debug(B.DBG_CAND)
    dec.close()

    def operand(a):
        return torch.from_numpy(np.ascontiguousarray(a)).double()
    r = h + torch.nn.functional.silu(h @ operand(w["medusa.0.w"]).T + operand(w["medusa.0.b"]))
    z = (r @ operand(w["lm_head"]).T).numpy()
    size = (r.abs() @ operand(w["lm_head"]).abs().T).numpy()
    for b in range(batch):
        got = cand[b, 1]
        assert len(set(got.tolist())) == kmax
        if classes:
            best = int(np.argmax(z[b, :classes]))
            assert got.tolist() == [best + classes * i for i in range(kmax)]
            continue
        tol = 4 * 256 * 2.0 ** -24 * size[b].max()   # (256 roundings of a sum here, and as many in r, on both sides of a comparison)
        picked = z[b][got]
        assert (np.diff(picked) <= tol).all()
        assert np.delete(z[b], got).max() <= picked[-1] + tol


@pytest.mark.parametrize("heads,hd,T,batch", [(1, 32, 20, 1), (1, 32, 29, 3), (4, 64, 16, 2)])
def test_row_maxima_have_room(heads, hd, T, batch):
    """The float32 argmax reads the row maxima that lm_head leaves, whatever the width of the queries."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="room", vocab=32016, d_ffn=704, n_heads=heads, n_kv_heads=heads, head_dim=hd, topk=(4, 2, 2), tree_nodes=T, seed=7)
    dec = SpecDecoder(cfg, upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, T), 64, max_batch=batch)
    dec.prefill([draw_prompt(cfg.with_(seed=30 + b), 5 + b) for b in range(batch)])
    dec.set_option(B.OPT_TRACE, 1)
    dec.step()
    ran = [r[0] for r in dec.trace()]
    dec.close()
    assert "topk_tiles" in ran and "argmax_tiles" in ran and "argmax_partials_tc" not in ran
