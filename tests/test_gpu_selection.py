"""Selection over the vocabulary: top-k lists with many equal logits, the argmax of many rows, sampling and typical
acceptance on vocabularies that are no multiple of a vector."""
import numpy as np
import pytest

from synthetic import draw_prompt, draw_weights, get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


@pytest.mark.parametrize("dtype,vocab,batch,period", [("bf16", 3000, 1, 1), ("bf16", 32016, 1, 1), ("bf16", 32016, 16, 1),
                                                      ("bf16", 2999, 2, 7), ("fp32", 3000, 1, 1), ("fp32", 1001, 2, 7)])
def test_top_k_and_argmax_with_equal_logits(torch, dtype, vocab, batch, period):
    """lm_head rows repeat with a period, so that every logit occurs vocab / period times: the lists are ordered by index
    among equals, rank t of a head is (best residue) + t * period, and every argmax lies in the first period."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="ties", dtype=dtype, vocab=vocab, d_ffn=704, n_heads=2, n_kv_heads=2, head_dim=128, topk=(10, 4, 2), tree_nodes=24, seed=3)
    w = draw_weights(cfg)
    w["lm_head"] = np.ascontiguousarray(w["lm_head"][np.arange(vocab) % period])
    dec = SpecDecoder(cfg, upload_weights(cfg, w), build_tree(cfg.topk, 24), 64, max_batch=batch)
    dec.prefill([draw_prompt(cfg, 5 + b) for b in range(batch)])
    dec.step()
    cand = dec.debug(B.DBG_CAND)
    first = cand[:, 1:, :1]
    assert (first < period).all()
    assert (cand[:, 1:] == first + period * np.arange(dec.kmax)).all()
    assert (dec.debug(B.DBG_ARGMAX) < period).all()
    dec.close()


@pytest.mark.parametrize("vocab", [1001, 3000])
def test_head_rows_in_several_passes(torch, vocab):
    """Without tensor cores the heads' logits share the verification pass's buffer: 24 (sequence, head) rows where it holds 16
    (or 15, padded to whole vectors) are selected from in two passes, with each sequence's own candidates."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="head_rows", vocab=vocab, seed=9)
    dw, tree = upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, 2)

    def candidates(prompts):
        dec = SpecDecoder(cfg, dw, tree, 64, max_batch=len(prompts))
        dec.prefill(prompts)
        dec.step()
        cand = dec.debug(B.DBG_CAND).copy()
        dec.close()
        return cand

    prompts = [draw_prompt(cfg.with_(seed=20 + b), 5 + b) for b in range(8)]
    together = candidates(prompts)
    for b, p in enumerate(prompts):
        assert np.array_equal(together[b], candidates([p])[0]), b


@pytest.mark.parametrize("vocab", [1001, 4096 * 8 + 4, 40003])
def test_sampled_decoding_vocabulary_sizes(torch, vocab):
    """Typical acceptance and sampling where the row does not fill a thread's share evenly: fewer tokens than threads, just
    past the cached part of a row, and a size that is no multiple of four."""
    from paper_2503_14153_b200 import build_tree
    from tests_lockstep import run_lockstep
    cfg = get_config("c0", name="vocab", vocab=vocab, seed=8)
    rep = run_lockstep(cfg, draw_weights(cfg), build_tree(cfg.topk, cfg.tree_nodes), draw_prompt(cfg), 24, 1e-4, 1e-2,
                       accept_mode=1, typ=(0.09, 0.3, float(np.float32(0.8))), sampling=True, seed=11)
    assert rep.steps > 0


@pytest.mark.parametrize("vocab,rows,batch", [(131, 33, 1), (2999, 64, 1), (4100, 128, 1), (131, 43, 3), (2999, 64, 4), (4100, 50, 6)])
def test_row_maxima_out_of_the_projection(torch, vocab, rows, batch):
    """lm_head compares its own tiles' tokens (up to 128 rows and more, vocabularies that fill no tile): every row's argmax is that of
    the kept logits, and the same without them."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="maxima", dtype="bf16", vocab=vocab, d_ffn=704, n_heads=2, n_kv_heads=2, head_dim=128, n_medusa=3, topk=(16, 8, 4),
                     tree_nodes=rows, seed=5)
    dw, tree = upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, rows)
    got = []
    for flags in (B.FLAG_KEEP_LOGITS, 0):
        dec = SpecDecoder(cfg, dw, tree, 64, max_batch=batch, flags=flags)
        dec.prefill([draw_prompt(cfg.with_(seed=30 + b), 5 + b) for b in range(batch)])
        dec.step()
        got.append(dec.debug(B.DBG_ARGMAX).copy())
        if flags:
            assert (dec.debug(B.DBG_LOGITS).argmax(-1) == got[0]).all()
        dec.close()
    assert (got[0] == got[1]).all()
