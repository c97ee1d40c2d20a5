"""Projection kernels at the sizes where a launch takes another shape, against 64-bit products."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


def check_linear(torch, M, N, K, ctas):
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator().manual_seed(M + N + K)
    x = torch.randn((M, K), generator=g).bfloat16().cuda()
    w = (torch.randn((N, K), generator=g) * 0.02).bfloat16().cuda()
    want = x.double() @ w.double().T
    y = spec_op_linear(x, w, ctas)
    # float32 sums of K products: K / 2 roundings of the running sum, each at most 2^-24 of the sum of the magnitudes
    bound = (K / 2 + 8) * 2.0 ** -24 * (x.double().abs() @ w.double().abs().T)
    assert ((y.double() - want).abs() <= bound).all()


@pytest.mark.parametrize("M,chunks", [(16, 5), (16, 6), (16, 12), (16, 13), (32, 11), (32, 12), (48, 9), (64, 4), (64, 9), (64, 10),
                                      (80, 4), (112, 7), (128, 3), (128, 8)])
def test_ring_depths(torch, M, chunks):
    """Grids of at most one CTA an SM get a stage for every K chunk of a CTA (`chunks`, here of a cluster of eight): the ring of which two fit an
    SM and one chunk more, the deepest ring full and run through again, and activation rows that fill the MMA's N only in part."""
    check_linear(torch, M, 1000, 8 * 64 * chunks, 128)


@pytest.mark.parametrize("mode,cluster", [(0, 8), (1, 3), (2, 2), (3, 1), (3, 2), (3, 3), (3, 4), (3, 6), (3, 8)])
def test_rings_leave_no_cluster_waiting(torch, mode, cluster):
    """A ring that fills an SM is taken as long as all clusters of the launch are on the chip at once with it, the one of which two fit an SM beyond, and the
    one of which three do for output and down projections alone."""
    import ctypes as C
    from paper_2503_14153_b200 import load_library
    lib, out = load_library(), (C.c_int32 * 2)()

    def launch(rows, tiles, chunks):
        assert lib.spec_debug_cluster_residency(mode, rows, tiles, cluster, chunks, out) == 0
        return list(out)
    for rows in (1, 16, 17, 64) + ((65, 128) if mode != 1 else ()):
        two_an_sm = 5 if rows <= 32 else (4 if rows <= 64 else 3)
        for tiles in range(1, 160 // cluster + 2):            # (16 chunks a CTA, of gate and up 32: more than the deepest ring has stages)
            stages, alone = launch(rows, tiles, 16 * cluster)
            assert (stages > two_an_sm) == (tiles <= alone), (rows, tiles, stages, alone)
        assert launch(rows, 296 // cluster, 4 * cluster)[0] == (4 if mode == 0 and rows <= 16 else two_an_sm)


@pytest.mark.parametrize("N,chunks", [(1920, 90), (2048, 90), (2304, 96), (2944, 70), (4480, 50), (6144, 36)])
@pytest.mark.parametrize("M", [16, 64, 128])
def test_more_clusters_than_fit_alone(torch, M, N, chunks):
    """Projections of 15 to 18 clusters of eight, 23 of six, 35 of four and 48 of three with runs longer than the short ring."""
    check_linear(torch, M, N, 64 * chunks, 296)


def random_decoder(torch, cfg, seed, max_seq):
    from paper_2503_14153_b200 import FLAG_KEEP_LOGITS, SpecDecoder, build_tree
    g = torch.Generator(device="cuda").manual_seed(seed)
    d, F, HD, KD = cfg.d_model, cfg.d_ffn, cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim

    def normal(rows, cols, std):
        return (torch.randn((rows, cols), generator=g, device="cuda") * std).bfloat16()

    w = {"embed": normal(cfg.vocab, d, 1.0), "lm_head": normal(cfg.vocab, d, 0.02), "final_norm": torch.ones(d, device="cuda")}
    for l in range(cfg.n_layers):
        p = f"layers.{l}."
        w.update({p + "wqkv": normal(HD + 2 * KD, d, d ** -0.5), p + "wo": normal(d, HD, HD ** -0.5), p + "w_gate": normal(F, d, d ** -0.5),
                  p + "w_up": normal(F, d, d ** -0.5), p + "w_down": normal(d, F, F ** -0.5),
                  p + "attn_norm": torch.ones(d, device="cuda"), p + "ffn_norm": torch.ones(d, device="cuda")})
    for k in range(cfg.n_medusa):
        w[f"medusa.{k}.w"] = normal(d, d, 0.01)
        w[f"medusa.{k}.b"] = normal(1, d, 0.02)[0].contiguous()
    return SpecDecoder(cfg, w, build_tree(cfg.topk, cfg.tree_nodes), max_seq, max_batch=cfg.batch, flags=FLAG_KEEP_LOGITS)


@pytest.mark.parametrize("d,ffn,T", [
    (512, 1344, 65), (512, 1344, 96), (512, 1344, 97), (512, 2304, 128),      # clusters of eight (the last: too many of them, the streamer serves)
    (512, 1920, 100), (1024, 2752, 69), (1024, 2752, 128),                    # eight again, six, two rounds
    (1280, 3200, 77), (1280, 3968, 113),                                      # five, four: a chunk more than stages
    (2048, 5248, 80), (2048, 7936, 66), (1024, 16000, 112),                   # three (11 chunks a CTA: the ring refilled), two, one
    (256, 640, 70),                                                           # a run a chunk, fewer CTAs than the cap
])
def test_gate_up_in_clusters_as_the_streamer(torch, d, ffn, T):
    """Gate, up and SwiGLU of 65 to 128 rows in one kernel: a layer's hidden rows, its cache and the logits are those of the weight streamer with the
    kernel behind it, bit for bit."""
    import numpy as np
    from paper_2503_14153_b200 import binding as B
    from synthetic import get_config
    cfg = get_config("c0", name="glu", n_layers=2, d_model=d, n_heads=d // 128, n_kv_heads=max(1, d // 256), head_dim=128, d_ffn=ffn, vocab=1000, dtype="bf16",
                     rope_base=1e6, n_medusa=4, topk=(10, 4, 2, 2), tree_nodes=T)
    prompt = np.random.default_rng(T).integers(0, 1000, 90).astype(np.int32)
    seen, launches = {}, {}
    for mask in (7, 5):
        gpu = random_decoder(torch, cfg, 5, 160)
        gpu.set_option(B.OPT_CLUSTER_EPILOGUE, mask)
        gpu.prefill(prompt)
        before = gpu.query(B.Q_KERNEL_LAUNCHES)
        out = [gpu.step() for _ in range(2)]
        launches[mask] = gpu.query(B.Q_KERNEL_LAUNCHES) - before
        seen[mask] = [np.concatenate([np.append(t[0, :n[0]], n[0]) for t, n in out]), gpu.debug(B.DBG_HIDDEN), gpu.debug(B.DBG_LOGITS), *gpu.read_kv(0, 1, 0, 90 + T)]
        gpu.close()
    assert launches[5] - launches[7] == (0 if ffn == 2304 else 2 * 2)         # a kernel less in each layer of both steps: the two paths are two
    assert np.isfinite(seen[7][1]).all() and np.abs(seen[7][1]).max() > 0.1
    for a, b in zip(seen[7], seen[5]):
        assert a.tobytes() == b.tobytes()


@pytest.mark.parametrize("M,N,K,ctas", [
    (1008, 11008, 512, 296), (1488, 5000, 256, 100),          # the last wave's tiles in halves, on 74 and on 50 pairs of SMs
    (592, 19008, 256, 296), (2032, 9700, 128, 296),           # in quarters, the last of them without rows; columns that are no multiple of a tile
    (2032, 4700, 2048, 296), (1040, 2600, 512, 40),           # tiles of 192 and of 208 rows, quarters of 16-row groups that do not divide
    (144, 19000, 128, 296),                                   # a single tile of fewer rows than 256
])
def test_tile_heights(torch, M, N, K, ctas):
    """Projections of many rows in tiles of other heights, and in slices of tiles."""
    check_linear(torch, M, N, K, ctas)


def test_rows_do_not_depend_on_the_tiles(torch):
    """The same prompt three times in a pass of 384 rows, sixteen times in one of 2048 and ten times in one of 1280: q/k/v, output, gate+up and down go through tiles of 16
    to 256 rows and through halves of tiles, and every sequence gets the same bits. (An inner dimension below 64 chunks: no tile is shared.)"""
    import numpy as np
    from paper_2503_14153_b200 import binding as B
    from synthetic import get_config
    prompt = np.random.default_rng(3).integers(0, 1000, 120).astype(np.int32)
    first = None
    for batch in (3, 16, 10):
        cfg = get_config("c0", name="tiles", n_layers=3, d_model=1024, n_heads=16, n_kv_heads=4, head_dim=64, d_ffn=2752, vocab=1000, dtype="bf16", rope_base=1e6,
                         n_medusa=4, topk=(10, 4, 2, 2), tree_nodes=4, batch=batch)
        gpu = random_decoder(torch, cfg, 9, 140)
        gpu.prefill([prompt] * batch)
        h = gpu.debug(B.DBG_H_LAST)
        kv = [np.stack(gpu.read_kv(b, l, 0, 120)) for b in (0, batch // 2, batch - 1) for l in (1, 2)]
        gpu.close()
        assert np.isfinite(h).all() and np.abs(h).max() > 0.1
        first = (h[0], kv[0], kv[1]) if first is None else first
        assert all((row == first[0]).all() for row in h)
        assert all((a == first[1 + i % 2]).all() for i, a in enumerate(kv))


@pytest.mark.parametrize("d,heads,kv,hd,ffn,n", [
    (512, 4, 4, 128, 1344, 129), (512, 8, 2, 64, 1344, 256),       # eight runs of gate+up; a row, and all, of the second chunk
    (1024, 16, 4, 64, 2752, 250), (1024, 8, 8, 128, 704, 145),     # six; more than eight: chunk by chunk
    (2048, 16, 16, 128, 5504, 200),                                # three CTAs to two tiles: runs of other lengths in every second tile
    (1024, 32, 8, 64, 5248, 177),                                  # three; heads enough for the attention to take several rows' blocks a CTA
])
def test_two_chunks_at_once(torch, d, heads, kv, hd, ffn, n):
    """A lone prompt of two chunks in one pass over the weights: first token, hidden state, cache and the steps that follow are those of its chunks one after
    the other (to which it goes without the many-row kernel), bit for bit."""
    import numpy as np
    from paper_2503_14153_b200 import binding as B
    from synthetic import get_config
    cfg = get_config("c0", name="two", n_layers=3, d_model=d, n_heads=heads, n_kv_heads=kv, head_dim=hd, d_ffn=ffn, vocab=1000, dtype="bf16", rope_base=1e6,
                     n_medusa=4, topk=(10, 4, 2, 2), tree_nodes=20)
    prompt = np.random.default_rng(n).integers(0, 1000, n).astype(np.int32)
    seen, launches = {}, {}
    for wide in (1, 0):
        gpu = random_decoder(torch, cfg, 5, n + 40)
        gpu.set_option(B.OPT_WIDE_GEMM, wide)
        before = gpu.query(B.Q_KERNEL_LAUNCHES)
        gpu.prefill(prompt)
        launches[wide] = gpu.query(B.Q_KERNEL_LAUNCHES) - before
        seen[wide] = [gpu.debug(B.DBG_NEXT_ROOT), gpu.debug(B.DBG_H_LAST)] + [a for l in range(3) for a in gpu.read_kv(0, l, 0, n)]
        for t, c in (gpu.step() for _ in range(2)):
            seen[wide].append(np.append(t[0, :c[0]], c[0]))
        gpu.close()
    assert launches[1] == launches[0] if ffn == 704 else launches[1] < 0.7 * launches[0]      # (one pass over the layers, not two)
    assert np.isfinite(seen[1][1]).all() and np.abs(seen[1][1]).max() > 0.1
    for a, b in zip(seen[1], seen[0]):
        assert a.tobytes() == b.tobytes()


@pytest.mark.parametrize("d,ffn,T,batch,kernel", [
    (1024, 2752, 69, 1, "gemm_glu"), (1024, 2752, 23, 3, "gemm_glu"), (512, 2304, 128, 1, "gemm_stream<128>"),
    (1024, 2752, 64, 1, "gemm_cluster<64,swiglu>"), (1024, 2752, 43, 3, "gemm_pair<swiglu>"),
])
def test_gate_up_kernel_name(torch, d, ffn, T, batch, kernel):
    """The kernel that a decoder names for a step's gate and up projections is the one that runs: the streamer alone leaves the SwiGLU to another."""
    import numpy as np
    from paper_2503_14153_b200 import binding as B
    from synthetic import get_config
    cfg = get_config("c0", name="names", n_layers=1, d_model=d, n_heads=d // 128, n_kv_heads=d // 128, head_dim=128, d_ffn=ffn, vocab=1000, dtype="bf16",
                     rope_base=1e6, n_medusa=4, topk=(10, 4, 2, 2), tree_nodes=T, batch=batch)
    gpu = random_decoder(torch, cfg, 5, 160)
    gpu.prefill([np.arange(20 + b, dtype=np.int32) for b in range(batch)])
    gpu.set_option(B.OPT_TRACE, 1)
    gpu.step()
    ran = [r[0] for r in gpu.trace()]
    assert gpu.gate_up_kernel_name() == kernel and gpu.query(B.Q_CLUSTER_GATE_UP) == (kernel[:8] in ("gemm_glu", "gemm_clu"))
    assert ("swiglu_reduce_tc" in ran) == (kernel[:8] == "gemm_str")
    gpu.close()
