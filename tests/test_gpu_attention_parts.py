"""Attention whose query rows go to several CTAs, against the oracle."""
import pytest

from synthetic import draw_prompt, draw_weights, get_config

pytestmark = pytest.mark.gpu

TOL_BF16, TIE_GAP = 2e-2, 1e-2


@pytest.mark.parametrize("heads,kv,hd,T,batch", [
    (32, 2, 64, 65, 1),       # five blocks of 16 rows on four CTAs of two, the last without rows
    (32, 4, 128, 100, 1),     # seven on four
    (32, 8, 64, 128, 1),      # eight on four
    (24, 2, 128, 112, 2),     # two sequences: seven on two CTAs of four
    (16, 2, 64, 40, 3),       # two key groups: three on two CTAs, the second half empty
    (16, 4, 64, 64, 3),       # four on two
])
def test_rows_in_several_ctas(heads, kv, hd, T, batch):
    """More (sequence, head, 16 rows) blocks than SMs, but few (sequence, head)s: a CTA takes some of the rows. Prompts of one and of two chunks."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from tests_lockstep import run_lockstep_batch
    cfg = get_config("c0", name="attn_parts", n_layers=2, d_model=256, d_ffn=704, vocab=3000, dtype="bf16", norm_gain="random", rope_base=1e6,
                     n_medusa=4, topk=(10, 4, 2, 2), n_heads=heads, n_kv_heads=kv, head_dim=hd, tree_nodes=T, seed=7 + T)
    w = draw_weights(cfg)
    prompts = [draw_prompt(cfg.with_(seed=60 + i), 150 - 50 * i) for i in range(batch)]
    tree = build_tree(cfg.topk, T)
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, 200, max_batch=batch, flags=B.FLAG_KEEP_LOGITS)
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, 200) for b in {0, batch - 1}}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 3, TOL_BF16, TIE_GAP)
    gpu.close()
    assert all(reps[b].steps == 3 for b in oracles)
