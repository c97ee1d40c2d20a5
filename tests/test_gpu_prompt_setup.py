"""What prompt processing sets up: tables, counters and the free part of the cache."""
import numpy as np
import pytest

from synthetic import get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,max_batch,rounds", [
    ("bf16", 1, [[300], [20], [170]]),                        # long, then short: what the first left is cleared; two chunks
    ("bf16", 3, [[100, 31, 260], [16, 5], [40, 50, 7]]),      # a sequence less, and again as many
    ("fp32", 2, [[90, 40], [12], [33, 60]]),
    ("bf16", 33, [[9] * 33, [30] * 20]),                      # more sequences than the tables by value hold
    ("bf16", 1, [[12400], [12300]]),                          # more chunks than they hold
])
def test_nothing_left_of_earlier_prompts(dtype, max_batch, rounds):
    """Prompts after other prompts and steps: first tokens, hidden states and steps as on a fresh context, and zeros in the cache from the page of the
    first free slot on."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from synthetic import draw_weights
    cfg = get_config("c0", name="setup", n_layers=2, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=704, vocab=1000, dtype=dtype, rope_base=1e6,
                     n_medusa=3, topk=(4, 2, 2), tree_nodes=9, seed=3)
    dw = upload_weights(cfg, draw_weights(cfg))
    tree = build_tree(cfg.topk, 9)
    room = max(max(r) for r in rounds) + 40
    rng = np.random.default_rng(1)

    def results(dec, prompts):
        dec.prefill(prompts)
        out = [dec.debug(B.DBG_NEXT_ROOT), dec.debug(B.DBG_H_LAST)]
        for b, p in enumerate(prompts):
            free = (len(p) + cfg.page_size - 1) // cfg.page_size * cfg.page_size
            for kv in dec.read_kv(b, 1, free, min(room, free + 400) - free):
                assert not kv.any()
        if len(prompts) < dec.max_batch:
            assert not any(kv.any() for kv in dec.read_kv(dec.max_batch - 1, 0, 0, min(room, 300)))
        for _ in range(2):
            t, n = dec.step()
            out += [n, np.where(np.arange(t.shape[1]) < n[:, None], t, -1)]
        return out

    used = SpecDecoder(cfg, dw, tree, room, max_batch=max_batch)
    for lens in rounds:
        prompts = [rng.integers(0, cfg.vocab, n).astype(np.int32) for n in lens]
        fresh = SpecDecoder(cfg, dw, tree, room, max_batch=max_batch)
        a, b = results(used, prompts), results(fresh, prompts)
        fresh.close()
        for x, y in zip(a, b):
            assert x.tobytes() == y.tobytes()
    used.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_nothing_left_of_failed_steps(dtype):
    """Steps that report an error (a candidate outside the vocabulary) move a sequence on all the same: the next prompt clears what all of them have
    written, not what the first one could have."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, SpecError, build_tree, upload_weights
    from synthetic import draw_weights
    cfg = get_config("c0", name="setup", n_layers=2, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=704, vocab=1000, dtype=dtype, rope_base=1e6,
                     n_medusa=3, topk=(4, 2, 2), tree_nodes=9, seed=3)
    dec = SpecDecoder(cfg, upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, 9), 400, max_batch=1)
    rng = np.random.default_rng(2)
    dec.prefill(rng.integers(0, cfg.vocab, 300).astype(np.int32))
    outside = np.full((1, cfg.n_medusa, dec.kmax), cfg.vocab, np.int32)
    for _ in range(40):
        with pytest.raises(SpecError):
            dec.step(outside)
    assert any(kv.any() for kv in dec.read_kv(0, 1, 336, 12))             # (beyond the page that a step at the prompt's end reaches)
    dec.prefill(rng.integers(0, cfg.vocab, 20).astype(np.int32))
    for kv in dec.read_kv(0, 1, 32, 368):
        assert not kv.any()
    dec.close()


def test_failed_prompt_waits_for_its_copies():
    """A prompt whose processing ends with an error on the host (here a lm_head that no tensor map takes, after the layers have been enqueued) is
    returned from when the stream is through: page-locked tokens are the caller's again."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from synthetic import draw_weights
    cfg = get_config("c0", name="setup", n_layers=2, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=704, vocab=1000, dtype="bf16", rope_base=1e6,
                     n_medusa=3, topk=(4, 2, 2), tree_nodes=9, seed=3)
    w = upload_weights(cfg, draw_weights(cfg))
    odd = torch.zeros(cfg.vocab * cfg.d_model + 1, dtype=torch.bfloat16, device="cuda")
    odd[1:] = w["lm_head"].reshape(-1)
    w["lm_head"] = odd[1:].view(cfg.vocab, cfg.d_model)                   # two bytes off the boundary
    dec = SpecDecoder(cfg, w, build_tree(cfg.topk, 9), 100, packed=False)
    tokens, offsets = torch.zeros(30, dtype=torch.int32).pin_memory(), np.array([0, 30], np.int32)
    a = torch.randn((8192, 8192), device="cuda").bfloat16()
    assert dec.lib.spec_prefill(dec._ctx, 1, tokens.data_ptr(), offsets.ctypes.data) != 0     # (a kernel's first launch loads it, which may wait by itself)
    a @ a
    torch.cuda.synchronize()
    for _ in range(60):                                                   # some 40 ms of work before the prompt's
        a @ a
    assert not dec.stream.query()
    assert dec.lib.spec_prefill(dec._ctx, 1, tokens.data_ptr(), offsets.ctypes.data) != 0
    assert dec.stream.query()
    dec.close()


def test_refused_prompts_leave_the_batch():
    """More prompts than the decoder has room for, or a prompt that is too long, are refused: steps and debug reads go on with the sequences that were there."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2503_14153_b200 import SpecDecoder, SpecError, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from synthetic import draw_weights
    cfg = get_config("c0", name="setup", n_layers=1, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=704, vocab=1000, n_medusa=3, topk=(4, 2, 2),
                     tree_nodes=9, seed=3)
    dec = SpecDecoder(cfg, upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, 9), 100, max_batch=3)
    prompts = [np.arange(20 + b, dtype=np.int32) for b in range(2)]
    dec.prefill(prompts)
    first = dec.debug(B.DBG_H_LAST)
    for refused in ([prompts[0]] * 4, [np.zeros(100, np.int32)] * 3):
        with pytest.raises(SpecError):
            dec.prefill(refused)
        assert np.array_equal(dec.debug(B.DBG_H_LAST), first)
        tokens, counts = dec.step() if len(refused) == 3 else (first, first)
        assert len(tokens) == len(counts) == 2
    dec.close()
