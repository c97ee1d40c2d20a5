"""Passes of more than 128 rows against the oracle: the two-SM projection kernel and its epilogues at the edges of
their tiles."""
import pytest

from synthetic import draw_prompt, draw_weights, get_config

pytestmark = pytest.mark.gpu

TOL_BF16, TIE_GAP = 2e-2, 1e-2
BASE = get_config("c0", name="many_rows", n_layers=2, d_model=256, d_ffn=704, vocab=3000, dtype="bf16", norm_gain="random",
                  rope_base=1e6, n_medusa=4, topk=(10, 4, 2, 2), tree_nodes=64)


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


@pytest.mark.parametrize("heads,kv,hd,ffn,T,batch", [
    (4, 2, 64, 704, 43, 3),       # 129 rows: the fewest; half a gate/up tile at the end, rotation pairs 32 lanes apart
    (2, 2, 128, 704, 47, 5),      # 235 rows: an activation tile that is not full, rotation pairs 64 lanes apart
    (6, 3, 64, 192, 64, 6),       # 384 rows: half of the second activation tile; weight tiles shared by nothing (odd counts)
    (4, 2, 64, 1344, 128, 4),     # 512 rows: two full activation tiles, grouped heads
])
def test_many_row_projections_vs_oracle(torch, heads, kv, hd, ffn, T, batch):
    """Batched verification with 129 to 512 rows: RoPE and the cache store, the residual add and SwiGLU all happen in the
    projection kernel's epilogue; logits, hidden and cache rows of two sequences against an oracle each."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from tests_lockstep import run_lockstep_batch
    cfg = BASE.with_(n_heads=heads, n_kv_heads=kv, head_dim=hd, d_ffn=ffn, tree_nodes=T, seed=41 + T)
    w = draw_weights(cfg)
    prompts = [draw_prompt(cfg.with_(seed=60 + i), 9 + 37 * i) for i in range(batch)]
    tree = build_tree(cfg.topk, T)
    room = max(len(p) for p in prompts) + 40
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, room, max_batch=batch, flags=B.FLAG_KEEP_LOGITS)
    assert gpu.query(B.Q_WIDE_GEMM) == 1
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, room) for b in (0, batch - 1)}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 3, TOL_BF16, TIE_GAP)
    gpu.close()
    for b in oracles:
        assert reps[b].steps == 3
