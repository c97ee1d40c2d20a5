"""Whole-valued outputs of the decode loop, pinned (needs a B200): the tokens of every step and how many were accepted.

The split of the inner dimension in a 16-bit layer decides how its results round, rounded results travel through all layers, and where
two candidates of an extra head lie close the order of the two decides at which step a token is accepted. A kernel that adds the same
products in another order is as close to the exact result and still moves some of these. The recorded runs are
long enough that such a change shows in several of them: golden/decode_streams.txt holds, for each run, the accepted lengths step by step and a
checksum of the emitted tokens.

The model is synthetic but peaked, as a trained one is: row t of lm_head is a sum of the embeddings of the tokens before t in a fixed cyclic
order, with falling weights, so that the heads' candidates are the tokens that follow and a step accepts two or three of them.
"""
import math
import os
import zlib

import numpy as np
import pytest

from synthetic import get_config

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "decode_streams.txt")
STRIDE = 977
LEVELS = [1.0] + [0.5 * 0.88 ** i for i in range(9)]
BASE = get_config("c0", name="peaked", n_layers=6, d_model=1024, n_heads=16, n_kv_heads=4, head_dim=64, d_ffn=2752, vocab=3000, dtype="bf16",
                  rope_base=1e6, n_medusa=4, topk=(10, 4, 2, 2), norm_gain="random", seed=300)

# name: (tree nodes, prompt lengths of a batch, batches)
RUNS = {
    "rows_16": (16, (100,), 60),
    "rows_23": (23, (100,), 60),
    "rows_64": (64, (100,), 60),
    "rows_100": (100, (100,), 60),
    "batch_3": (23, (37, 224, 411), 40),
}
STEPS = 16


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def draw_peaked(torch, cfg):
    """Device tensors in the layout the decoder takes, drawn with numpy."""
    d, F, V, L, D = cfg.d_model, cfg.d_ffn, cfg.vocab, cfg.n_layers, cfg.head_dim
    rng = np.random.default_rng(np.random.SeedSequence([cfg.seed, 7]))

    def normal(rows, cols, std):
        a = rng.standard_normal((rows, cols), dtype=np.float32)
        a *= np.float32(std)
        return torch.from_numpy(a).bfloat16().cuda()

    def gain():
        return torch.from_numpy((1.0 + 0.1 * rng.standard_normal(d, dtype=np.float32)).astype(np.float32)).cuda()

    w = {"embed": normal(V, d, 1.0)}
    head = np.zeros((V, d), dtype=np.float32)
    embed = w["embed"].float().cpu().numpy()
    for i, a in enumerate(LEVELS):
        head += np.float32(0.02 * a) * np.roll(embed, STRIDE * (i + 1), 0)
    w["lm_head"] = torch.from_numpy(head).bfloat16().cuda()
    w["final_norm"] = gain()
    wide = math.sqrt(4096 / d)
    in_std, out_std = 0.02 * wide, 0.02 / math.sqrt(2 * L) * wide
    for l in range(L):
        p = f"layers.{l}."
        w[p + "wqkv"] = normal((cfg.n_heads + 2 * cfg.n_kv_heads) * D, d, in_std)
        w[p + "wo"] = normal(d, cfg.n_heads * D, out_std)
        w[p + "w_gate"], w[p + "w_up"], w[p + "w_down"] = normal(F, d, in_std), normal(F, d, in_std), normal(d, F, out_std)
        w[p + "attn_norm"], w[p + "ffn_norm"] = gain(), gain()
    for k in range(cfg.n_medusa):
        w[f"medusa.{k}.w"] = normal(d, d, in_std / 2)
        w[f"medusa.{k}.b"] = normal(1, d, 0.02)[0].contiguous()
    return w


def recorded(torch, weights, name):
    """One line a batch of prompts: accepted lengths (a digit a step, sequences separated by commas), checksum of the tokens."""
    from paper_2503_14153_b200 import SpecDecoder, build_tree
    nodes, lens, batches = RUNS[name]
    cfg = BASE.with_(tree_nodes=nodes)
    dec = SpecDecoder(cfg, weights, build_tree(cfg.topk, nodes), max(lens) + 5 * (STEPS + 1), max_batch=len(lens))
    out = []
    for k in range(batches):
        rng = np.random.default_rng(np.random.SeedSequence([cfg.seed, 8, k]))
        dec.prefill([rng.integers(0, cfg.vocab, n).astype(np.int32) for n in lens])
        counts, crc = [], 0
        for _ in range(STEPS):
            t, n = dec.step()
            counts.append(n.copy())
            for b in range(len(lens)):
                crc = zlib.crc32(np.ascontiguousarray(t[b, :n[b]], dtype="<i4").tobytes(), crc)
        out.append(f"{name} {k} {','.join(''.join(str(c[b]) for c in counts) for b in range(len(lens)))} {crc:08x}")
    dec.close()
    return out


@pytest.fixture(scope="module")
def weights(torch):
    return draw_peaked(torch, BASE)


@pytest.mark.parametrize("name", list(RUNS))
def test_tokens_and_accepted_lengths_as_recorded(torch, weights, name):
    with open(GOLDEN) as f:
        want = [line.strip() for line in f if line.split(" ")[0] == name]
    got = recorded(torch, weights, name)
    assert len(want) == RUNS[name][2]
    assert got == want, [(g, w) for g, w in zip(got, want) if g != w]
