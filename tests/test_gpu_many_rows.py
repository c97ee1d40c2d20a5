"""Passes of more than 128 rows against the oracle: the two-SM projection kernel and its epilogues at the edges of
their tiles."""
import numpy as np
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


@pytest.mark.parametrize("d,heads,kv,hd,ffn,T,batch", [
    # d 4096: q/k/v in 3 tiles of 4 parts each (heads of 128) and in 2 of 4 (heads of 64), gate/up in 2 tiles of 4, 129 rows
    (4096, 2, 2, 128, 256, 43, 3), (4096, 4, 2, 64, 128, 43, 3),
    # grouped heads at 256 rows: q/k/v in 24 tiles of 3, output in 16 of 4, gate/up in 32 of 2, down in 16 of 4
    (4096, 32, 8, 128, 4096, 64, 4),
    # 768 rows: down in 24 tiles of 3; 320 rows, the second activation tile a quarter full: down in 16 tiles of 4
    (2048, 4, 2, 64, 4096, 128, 6), (2048, 4, 2, 64, 4160, 64, 5),
    # an inner dimension of 8192 and few tiles: down in 2 tiles of 8; the output projection (4096) in 2 of 4
    (256, 32, 2, 128, 8192, 60, 5),
])
def test_shared_tiles_vs_oracle(torch, d, heads, kv, hd, ffn, T, batch):
    """Projections with tiles for less than half of the CTA pairs and an inner dimension of 4096 or more: the K chunks of a tile
    are shared between clusters, and the last to arrive adds the parts and does the tile's epilogue. Three steps in a
    row also show that the arrival counters are back at zero."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from tests_lockstep import run_lockstep_batch
    cfg = BASE.with_(n_layers=1, d_model=d, n_heads=heads, n_kv_heads=kv, head_dim=hd, d_ffn=ffn, n_medusa=2, topk=(10, 16), tree_nodes=T,
                     seed=91 + T)
    w = draw_weights(cfg)
    prompts = [draw_prompt(cfg.with_(seed=60 + i), 9 + 37 * i) for i in range(batch)]
    tree = build_tree(cfg.topk, T)
    room = max(len(p) for p in prompts) + 40
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, room, max_batch=batch, flags=B.FLAG_KEEP_LOGITS)
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, room) for b in (0, batch - 1)}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 3, TOL_BF16, TIE_GAP, tie_from_row_error=True)
    gpu.close()
    for b in oracles:
        assert reps[b].steps == 3


@pytest.mark.parametrize("hd,lengths", [
    (128, (2500,)),               # 20 chunks of one prompt: two passes, the second sees the first pass's chunks in the cache
    (64, (1300,)),                # 11 chunks in one pass, the mma.sync attention
    (128, (300, 5, 129, 700)),    # chunks of several prompts in a pass, last chunks of 44, 5, 1 and 60 rows
    (64, (17, 33)),               # short prompts: a chunk each that is mostly empty
])
def test_prompts_in_chunks_vs_oracle(torch, hd, lengths):
    """Prompt processing deals the 128-token chunks of all prompts to shared passes: the first root, the hidden state and
    the cache rows after it, and two steps on top, against an oracle for each prompt."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from tests_lockstep import run_lockstep_batch
    from paper_2503_14153_b200 import binding as B
    cfg = BASE.with_(n_heads=4, n_kv_heads=2, head_dim=hd, tree_nodes=32, seed=51)
    w = draw_weights(cfg)
    prompts = [draw_prompt(cfg.with_(seed=70 + i), n) for i, n in enumerate(lengths)]
    tree = build_tree(cfg.topk, 32)
    room = max(lengths) + 40
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, room, max_batch=len(lengths), flags=B.FLAG_KEEP_LOGITS)
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, room) for b in range(len(lengths))}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 2, TOL_BF16, TIE_GAP)
    gpu.close()
    for b in oracles:
        assert reps[b].steps == 2


@pytest.mark.parametrize("hd,lengths,nbytes", [(128, (1300,), 18661376), (64, (300, 5, 129, 700), 44637184)])
def test_prompts_in_a_smaller_workspace(torch, monkeypatch, hd, lengths, nbytes):
    """A workspace that holds the activations of one chunk a sequence and no more (the sizes that sufficed when a pass took no
    more than that) is accepted and gives the same tokens; one that does not even hold those is refused."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from tests_lockstep import run_lockstep_batch
    from paper_2503_14153_b200 import binding as B
    cfg = BASE.with_(n_heads=4, n_kv_heads=2, head_dim=hd, tree_nodes=32, seed=51)
    w = draw_weights(cfg)
    dw = upload_weights(cfg, w)
    prompts = [draw_prompt(cfg.with_(seed=70 + i), n) for i, n in enumerate(lengths)]
    tree = build_tree(cfg.topk, 32)
    room = max(lengths) + 40
    size = {"n": nbytes}
    monkeypatch.setattr(B.load_library(), "spec_workspace_bytes", lambda *a: size["n"])
    gpu = SpecDecoder(cfg, dw, tree, room, max_batch=len(lengths), flags=B.FLAG_KEEP_LOGITS)
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, room) for b in range(len(lengths))}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 2, TOL_BF16, TIE_GAP)
    gpu.close()
    for b in oracles:
        assert reps[b].steps == 2
    size["n"] = nbytes // 2
    with pytest.raises(B.SpecError, match="workspace too small"):
        SpecDecoder(cfg, dw, tree, room, max_batch=len(lengths), flags=B.FLAG_KEEP_LOGITS)


@pytest.mark.parametrize("M,N,K,ctas", [(144, 128, 64, 1), (272, 300, 64, 2), (1008, 1000, 704, 148), (2048, 129, 128, 296),
                                        (512, 4096, 4096, 7),
                                        (256, 4096, 4096, 296), (272, 300, 8192, 296), (512, 5000, 4096, 296),
                                        (1008, 11008, 4096, 296),
                                        # fewer CTAs, so that these have two tiles a CTA and take the two-SM kernel too: halves of
                                        # one chunk of the inner dimension and of 5 and 6, a tile a cluster, a long inner dimension
                                        (2048, 129, 128, 16), (1008, 1000, 704, 30), (512, 5000, 4096, 80), (1536, 300, 8192, 16)])
def test_op_linear_many_rows(torch, M, N, K, ctas):
    """More than 128 rows of the stand-alone projection, on the two-SM kernel where a CTA has two (128 x 128) tiles or more, on
    the weight-streaming kernel otherwise: one weight tile (computed by both SMs of a pair, stored once), ragged columns
    and activation tiles, more tiles than CTA pairs. Bound: K accumulations in float32, each off by at most one
    unit in the last place of the running sum, against sum |x w|."""
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator(device="cuda").manual_seed(M + N)
    x = torch.randn((M, K), generator=g, device="cuda", dtype=torch.bfloat16)
    w = torch.randn((N, K), generator=g, device="cuda", dtype=torch.bfloat16)
    y = spec_op_linear(x, w, ctas)
    want, size = x.double() @ w.double().T, x.double().abs() @ w.double().abs().T
    assert ((y.double() - want).abs() <= K * 2.0 ** -23 * size).all()
    # the bound above is loose where K is large: a dropped or doubled 64-wide chunk would still show here
    assert ((y.double() - want).norm() / want.norm()).item() < 2e-5


@pytest.mark.parametrize("M,N,K,streamed", [(1008, 11008, 4096, 3.88e-6), (1536, 12000, 11008, 1.150e-5), (2048, 11008, 1024, 9.35e-7),
                                            (2048, 12000, 256, 2.17e-7), (1536, 12000, 128, 1.113e-7)])
def test_op_linear_many_rows_error(torch, M, N, K, streamed):
    """Whole tiles are no further from the 64-bit product than the weight-streaming kernel was at these shapes (`streamed`,
    measured on random normal operands; it moves by less than 0.5% with the seed)."""
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn((M, K), generator=g, device="cuda", dtype=torch.bfloat16)
    w = torch.randn((N, K), generator=g, device="cuda", dtype=torch.bfloat16)
    y = spec_op_linear(x, w).double()
    want = x.double() @ w.double().T
    assert ((y - want).norm() / want.norm()).item() <= 1.005 * streamed


@pytest.mark.parametrize("lens,layers,hd,batch", [
    ([129], 2, 128, 1),             # two chunks in two passes: the first ends no prompt
    ([256], 1, 64, 1),              # the only layer is the last one; the last row of a chunk
    ([300], 2, 128, 1),             # one pass of three chunks
    ([384, 1, 130, 128], 2, 64, 5), # ragged, a prompt of one token, whole chunks, a free sequence
    ([2400, 7], 1, 128, 2),         # 20 chunks: the first pass ends no prompt, the second both
])
def test_last_layer_of_a_prompt_for_its_last_rows(torch, lens, layers, hd, batch):
    """Prompt processing takes only the prompts' last tokens through the rest of the last layer: first token, hidden state, cache rows of
    the whole prompts and the steps that follow against an oracle each. A second, shorter set of prompts in the same context finds
    the slots behind it cleared."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from tests_lockstep import run_lockstep_batch
    cfg = BASE.with_(n_layers=layers, d_model=512, n_heads=512 // hd, n_kv_heads=512 // hd, head_dim=hd, d_ffn=1344, tree_nodes=16, seed=130 + len(lens))
    w = draw_weights(cfg)
    tree = build_tree(cfg.topk, 16)
    room = max(lens) + 40
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, room, max_batch=batch, flags=B.FLAG_KEEP_LOGITS)
    model = OracleModel(cfg, w)
    for k, sizes in enumerate((lens, [max(1, n // 2) for n in reversed(lens)])):
        prompts = [draw_prompt(cfg.with_(seed=150 + 10 * k + i), n) for i, n in enumerate(sizes)]
        oracles = {b: OracleSpecDecoder(model, tree, room) for b in {0, len(sizes) - 1}}
        reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 2, TOL_BF16, TIE_GAP, tie_from_row_error=True)
        for b in oracles:
            assert reps[b].steps == 2
        k0, v0 = gpu.read_kv(0, layers - 1, len(prompts[0]) + 30, 2)
        assert not k0.any() and not v0.any()          # nothing was written there since the prompts were processed
    gpu.close()


@pytest.mark.parametrize("lens,hd,kv,d,ffn", [
    ([300], 128, 4, 512, 1344),                      # one pass, shared K/V attention by key splits
    ([300], 64, 2, 512, 4160),                       # the down projection's tiles are shared between clusters
    ([129, 256, 1, 700, 128], 64, 8, 512, 1344),     # ragged: chunks of one row, whole chunks, a lone token
    ([1600, 40], 128, 1, 512, 1344),                 # longer than 512 positions
    ([200, 333, 520, 77, 900, 64], 128, 8, 1024, 1344),
    ([2400, 7], 128, 4, 512, 1344),                  # two passes, the first of which ends no prompt
    ([256, 129], 128, 32, 4096, 1344),               # query, key and value tiles shared or not by how many there are in all
    ([250] * 140, 64, 2, 512, 704),                  # more last rows than an activation tile's half, in several passes
])
def test_last_rows_as_in_the_whole_layer(torch, lens, hd, kv, d, ffn):
    """The last layer goes on with the prompts' last rows alone, with the sums of the whole layer bit for bit: with a layer behind it
    that adds nothing (output and down projections of zeros) it is computed for all rows. Hidden states, first tokens, keys and values."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    heads = d // hd
    two = BASE.with_(n_layers=2, d_model=d, n_heads=heads, n_kv_heads=kv, head_dim=hd, d_ffn=ffn, vocab=1000, tree_nodes=4, seed=170 + len(lens) + ffn)
    w = draw_weights(two)
    w["layers.1.wo"][:] = 0
    w["layers.1.w_down"][:] = 0
    prompts = [draw_prompt(two.with_(seed=180 + i), n) for i, n in enumerate(lens)]
    got = []
    for cfg in (two.with_(n_layers=1), two):
        dec = SpecDecoder(cfg, upload_weights(cfg, {k: v for k, v in w.items() if cfg.n_layers == 2 or not k.startswith("layers.1.")}),
                          build_tree(cfg.topk, 4), max(lens) + 20, max_batch=len(lens))
        dec.prefill(prompts)
        last = len(lens) - 1
        got.append([dec.debug(B.DBG_H_LAST).copy(), dec.debug(B.DBG_NEXT_ROOT).copy(), dec.debug(B.DBG_SEQLEN).copy(),
                    *dec.read_kv(0, 0, 0, lens[0]), *dec.read_kv(last, 0, 0, lens[last])])
        dec.close()
    for one, whole in zip(*got):
        assert np.array_equal(one, whole), int((one != whole).sum())


@pytest.mark.parametrize("T,heads,kv,batch", [(48, 16, 4, 12), (64, 32, 32, 5), (80, 16, 16, 11), (128, 32, 8, 6)])
def test_attention_items_one_after_another(torch, T, heads, kv, batch):
    """Batched passes with more (sequence, head) items than SMs (160 to 192): a CTA of the tcgen05 attention takes several, of one to four
    key tiles each, so that an item's first tile falls to either softmax group; 64 and 128 rows a CTA, grouped heads. Two
    sequences against an oracle each; two steps show that the item counter is back at zero."""
    from oracle.decoder import OracleModel
    from oracle.spec import OracleSpecDecoder
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    from tests_lockstep import run_lockstep_batch
    cfg = BASE.with_(n_heads=heads, n_kv_heads=kv, head_dim=128, tree_nodes=T, seed=210 + T)
    w = draw_weights(cfg)
    prompts = [draw_prompt(cfg.with_(seed=220 + i), 3 + (97 * i) % 389) for i in range(batch)]
    tree = build_tree(cfg.topk, T)
    room = max(len(p) for p in prompts) + 40
    gpu = SpecDecoder(cfg, upload_weights(cfg, w), tree, room, max_batch=batch, flags=B.FLAG_KEEP_LOGITS)
    gpu.set_option(B.OPT_LONG_ATTN_KEYS, 1)
    model = OracleModel(cfg, w)
    oracles = {b: OracleSpecDecoder(model, tree, room) for b in (1, batch - 1)}
    reps = run_lockstep_batch(cfg, gpu, oracles, prompts, 2, TOL_BF16, TIE_GAP, tie_from_row_error=True)
    gpu.close()
    for b in oracles:
        assert reps[b].steps == 2


@pytest.mark.parametrize("T,prompt", [(64, 300), (33, 200), (128, 200), (80, 500)])
def test_attention_does_not_depend_on_the_place_in_a_batch(torch, T, prompt):
    """Twelve times the same prompt, 192 (sequence, head) items on the SMs: a CTA's second item begins with an odd tile here (three or
    five tiles an item), that is, with the other softmax group. Prompt processing and two steps give every sequence the same bits."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = BASE.with_(n_heads=16, n_kv_heads=4, head_dim=128, tree_nodes=T, seed=240 + T)
    dec = SpecDecoder(cfg, upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, T), prompt + 40, max_batch=12)
    dec.set_option(B.OPT_LONG_ATTN_KEYS, 1)
    dec.prefill([draw_prompt(cfg, prompt)] * 12)

    def same(a):
        return (a == a[:1]).all()
    assert same(dec.debug(B.DBG_H_LAST))
    for b in (0, 11):
        k, v = dec.read_kv(b, 1, 0, prompt)
        first = (k.copy(), v.copy()) if b == 0 else first
    assert (first[0] == k).all() and (first[1] == v).all()
    for _ in range(2):
        toks, counts = dec.step()
        assert same(counts) and same(toks[:, :counts[0]])
        assert same(dec.debug(B.DBG_HIDDEN).reshape(12, T, -1)) and same(dec.debug(B.DBG_H_LAST))
    dec.close()


@pytest.mark.parametrize("T", [64, 100])
def test_a_sequence_without_room_leaves_the_others_alone(torch, T):
    """192 (sequence, head) items, and the longest sequence, with whose items sixteen CTAs begin and whose first tiles they have asked for,
    turns out to be beyond its cache (its length on the device is set so): the step says so, and the other eleven sequences
    get the bits of an undisturbed decoder."""
    from paper_2503_14153_b200 import SpecDecoder, SpecError, build_tree, upload_weights
    from paper_2503_14153_b200 import binding as B
    cfg = BASE.with_(n_heads=16, n_kv_heads=4, head_dim=128, tree_nodes=T, seed=250 + T)
    dw, tree = upload_weights(cfg, draw_weights(cfg)), build_tree(cfg.topk, T)
    prompts = [draw_prompt(cfg.with_(seed=260 + i), 420 if i == 3 else 200 + 10 * i) for i in range(12)]
    got = []
    for disturbed in (False, True):
        dec = SpecDecoder(cfg, dw, tree, 480, max_batch=12)
        dec.set_option(B.OPT_LONG_ATTN_KEYS, 1)
        dec.prefill(prompts)
        if disturbed:
            # (the committed lengths lie behind the status word at the start of the workspace)
            start = (dec.workspace.data_ptr() + 1023) // 1024 * 1024 - dec.workspace.data_ptr()
            lengths = dec.workspace[start + 16:start + 16 + 48].view(torch.int32)
            assert lengths.tolist() == [len(p) for p in prompts]
            lengths[3] = 100000
            with pytest.raises(SpecError) as ei:
                dec.step()
            assert ei.value.code == -4, ei.value                  # SPEC_E_SEQLEN
        else:
            dec.step()
        got.append(dec.debug(B.DBG_HIDDEN).reshape(12, T, -1)[[b for b in range(12) if b != 3]].copy())
        dec.close()
    assert np.array_equal(*got)
