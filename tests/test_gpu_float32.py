"""The float32 kernels at the edges of their tiles: projections (split inner dimension, ragged rows and columns) and
attention (every head width, one tile of keys and several)."""
import pytest

from synthetic import draw_prompt, draw_weights, get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 8),           # one output, most lanes without a piece of the inner dimension
    (7, 301, 96),        # ragged rows and columns, less than one step of 128
    (3, 9, 2048),        # four warps split the inner dimension
    (9, 130, 264),       # two warps split it, the last step is not full
    (16, 32016, 256),    # a CTA's warps walk over the outputs, two row groups beside each other
    (100, 3000, 1024),   # 13 row groups
])
def test_op_linear_f32(torch, M, N, K):
    """Bound: K accumulations in float32, each off by at most half a unit in the last place of the running sum."""
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    x, w = torch.randn((M, K), generator=g, device="cuda"), torch.randn((N, K), generator=g, device="cuda")
    y = spec_op_linear(x, w)
    want, size = x.double() @ w.double().T, x.double().abs() @ w.double().abs().T
    assert ((y.double() - want).abs() <= K * 2.0 ** -24 * size).all()


@pytest.mark.parametrize("N,K", [(768, 256), (1000, 1024), (3000, 1024), (256, 688), (130, 264)])
def test_rows_do_not_depend_on_the_number_of_rows(torch, N, K):
    """A row's float32 sums are the same, bit for bit, whatever other rows the call has."""
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator(device="cuda").manual_seed(N + K)
    x, w = torch.randn((300, K), generator=g, device="cuda"), torch.randn((N, K), generator=g, device="cuda")
    whole = spec_op_linear(x, w)
    for m in (1, 4, 16, 33, 128):
        assert torch.equal(spec_op_linear(x[:m].contiguous(), w), whole[:m]), m


@pytest.mark.parametrize("N,K", [(1, 8), (37, 64), (3001, 128), (2999, 200), (3000, 256), (9600, 248)])
def test_activations_in_registers(torch, N, K):
    """Projections of an inner dimension of up to 256, whose warps keep their rows in registers: against 64 bits within the bound of K
    roundings, whatever the rows beside a row."""
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator(device="cuda").manual_seed(N + K)
    x, w = torch.randn((101, K), generator=g, device="cuda"), torch.randn((N, K), generator=g, device="cuda")
    whole = spec_op_linear(x, w)
    want, size = x.double() @ w.double().T, x.double().abs() @ w.double().abs().T
    assert ((whole.double() - want).abs() <= K * 2.0 ** -24 * size).all()
    for m in (1, 3, 4, 5, 8, 9, 17, 40):
        assert torch.equal(spec_op_linear(x[:m].contiguous(), w), whole[:m]), m


@pytest.mark.parametrize("hd,heads,kv,prompt_len,dtype", [
    (32, 4, 4, 150, "fp32"), (64, 4, 2, 140, "fp32"), (96, 2, 2, 70, "fp32"), (128, 2, 1, 63, "fp32"), (160, 2, 2, 33, "fp32"),
    (256, 2, 2, 100, "fp32"), (256, 1, 1, 1, "fp32"), (64, 4, 2, 140, "bf16"),
])
def test_plain_attention_vs_oracle(torch, hd, heads, kv, prompt_len, dtype):
    """Decoding on the CUDA-core kernels (bf16: the debug mode of the 16-bit path) with contexts of one key tile, several, and
    a last group of keys that is not full, grouped heads among them."""
    from paper_2503_14153_b200 import FLAG_SIMPLE_KERNELS, build_tree
    from tests_lockstep import run_lockstep
    cfg = get_config("c0", name="plain", n_heads=heads, n_kv_heads=kv, head_dim=hd, dtype=dtype, vocab=2000, seed=hd, norm_gain="random")
    rep = run_lockstep(cfg, draw_weights(cfg), build_tree(cfg.topk, cfg.tree_nodes), draw_prompt(cfg, prompt_len), 10,
                       1e-4 if dtype == "fp32" else 2e-2, 1e-2, flags=FLAG_SIMPLE_KERNELS if dtype == "bf16" else 0)
    assert rep.steps > 0


@pytest.mark.parametrize("hd,heads,kv,nodes", [(32, 4, 4, 1), (64, 4, 2, 7), (96, 2, 2, 29), (64, 8, 8, 64), (64, 8, 4, 100), (256, 2, 1, 16)])
def test_warps_of_a_row_vs_oracle(torch, hd, heads, kv, nodes):
    """Trees whose rows get several warps each in the CUDA-core attention (an odd number of rows among them, more warps than groups of
    keys or dimensions) and trees beyond that."""
    from paper_2503_14153_b200 import build_tree
    from tests_lockstep import run_lockstep
    cfg = get_config("c0", name="plain", n_heads=heads, n_kv_heads=kv, head_dim=hd, dtype="fp32", vocab=2000, seed=hd, norm_gain="random",
                     topk=(4, 2, 2) if nodes <= 29 else (10, 4, 2, 2), n_medusa=3 if nodes <= 29 else 4)
    rep = run_lockstep(cfg, draw_weights(cfg), build_tree(cfg.topk, nodes), draw_prompt(cfg, 50), 8, 1e-4, 1e-2)
    assert rep.steps > 0


@pytest.mark.parametrize("hd,heads,kv", [(32, 4, 2), (64, 4, 4), (160, 2, 1)])
def test_rows_of_ragged_prompts(torch, hd, heads, kv):
    """Queries, keys and values out of one projection for prompts that leave rows of the pass empty: every prompt as by itself, bit for bit."""
    import numpy as np
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = get_config("c0", name="ragged", n_heads=heads, n_kv_heads=kv, head_dim=hd, vocab=2000, seed=hd, norm_gain="random")
    w = upload_weights(cfg, draw_weights(cfg))
    prompts = [draw_prompt(cfg.with_(seed=40 + i), n) for i, n in enumerate((1, 37, 150))]

    def run(ps):
        dec = SpecDecoder(cfg, w, build_tree(cfg.topk, cfg.tree_nodes), 256, max_batch=len(ps))
        dec.prefill(ps)
        for _ in range(3):
            dec.step()
        h = np.array(dec.debug(B.DBG_H_LAST))
        dec.close()
        return h
    together = run(prompts)
    for i, p in enumerate(prompts):
        assert np.array_equal(run([p])[0], together[i]), i
