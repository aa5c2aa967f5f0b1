"""GPU tests at the sizes where a kernel's tiling or its dispatch changes: tile edges, remainders, ends of the range."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_2609_24197_b200 as m
    from paper_2609_24197_b200 import build
    build.build()
    m.load_library()
    return m


def _rand(shape, seed, dtype=torch.float16, std=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda") * std).to(dtype)


# rows that make the 2-SM kernel take tiles of many widths, full and with a remainder, whole waves and tail waves with one to eight slices (as
# asserted: rows per tile, slices, tiles, tiles of the last wave); weight rows that end inside a tile of the pair; more activation tiles (29) than
# one group of the walk holds
@pytest.mark.parametrize("M,n_out,K,tiles", [(256, 256, 64, (128, 1, 2, 2)), (257, 300, 520, (96, 1, 6, 6)), (289, 1000, 512, (112, 1, 12, 12)),
                                             (430, 2048, 1024, (112, 1, 32, 32)), (448, 2048, 1024, (112, 1, 32, 32)), (449, 512, 2048, (128, 4, 8, 8)),
                                             (549, 4096, 1024, (144, 1, 64, 64)), (640, 19200, 256, (224, 1, 225, 3)), (1153, 1111, 264, (128, 1, 50, 50)),
                                             (4500, 1200, 2048, (160, 1, 145, 71)), (270, 4096, 4096, (144, 2, 32, 32)), (257, 2560, 4096, (144, 3, 20, 20)),
                                             (130, 1024, 8192, (80, 8, 8, 8)), (1130, 4096, 4096, (240, 8, 80, 6))])
@pytest.mark.parametrize("kind", ["f32", "accumulate", "f16"])
def test_many_row_gemm_tile_widths(hs, M, n_out, K, tiles, kind):
    assert hs.hspec_debug_gemm_tiles(M, n_out, K) == tiles
    _gemm_against_fp64(hs, M, n_out, K, kind)


def _gemm_against_fp64(hs, M, n_out, K, kind):
    x, w = _rand((M, K), 1), _rand((n_out, K), 2, std=0.05)
    ref = x.double() @ w.double().t()
    y = torch.zeros((M, n_out), dtype=torch.float16 if kind == "f16" else torch.float32, device="cuda")
    if kind == "accumulate":
        y = _rand((M, n_out), 3, torch.float32)
        ref = ref + y.double()
    ws = torch.empty(hs.hspec_gemm_workspace_bytes(M, n_out, K), dtype=torch.uint8, device="cuda")
    hs.hspec_op_gemm(x, w, y, accumulate=kind == "accumulate", workspace=ws)
    # products of 16-bit values are exact in fp32; K additions of terms of size |x||w| round to 2^-24 of the running sum each
    # (bounded by the sum of magnitudes), the fp16 store to 2^-11 of the value
    mag = x.double().abs() @ w.double().abs().t() + ref.abs()
    bound = K * 2.0 ** -24 * mag + (2.0 ** -11 * ref.abs() + 1e-7 if kind == "f16" else 0.0)
    worst = float(((y.double() - ref).abs() / bound).max())
    assert worst <= 1.0, worst


# requests at the edges of the one-launch form's column chunks (32 per epilogue-warp chunk, 16 per MMA step) and of its range (128);
# vocabularies of less than a tile, of a tile and a row, and of more tiles than SMs; ranks below, at and above a 64-column box
@pytest.mark.parametrize("B,k,Vd,r", [(1, 1, 100, 8), (16, 3, 129, 64), (17, 4, 128, 72), (32, 2, 5000, 256), (33, 5, 19200, 256),
                                      (64, 3, 257, 136), (65, 2, 40000, 256), (96, 4, 3001, 256), (97, 2, 900, 512), (100, 3, 41000, 256), (112, 3, 700, 64), (113, 3, 700, 64), (128, 5, 21000, 256),
                                      (129, 2, 300, 64)])
@pytest.mark.parametrize("write", [True, False])
def test_markov_head_chunks_and_tiles(hs, B, k, Vd, r, write):
    g = torch.Generator().manual_seed(B * 1000 + k)
    # logits on a grid of 2^-6 and factors on a grid of 2^-4 with |x| <= 1/2: every product and sum below is exact in fp32, so the
    # ids (planted and natural ties included, lowest index first) and the logits must match exactly
    logits = torch.randint(-256, 257, (B * k, Vd), generator=g).float() / 64
    logits[:, Vd // 2] = logits.max() + 1
    logits[:, Vd // 3] = logits[:, Vd // 2]
    W_in = (torch.randint(-8, 9, (Vd, r), generator=g).float() / 16).half()
    W_out = (torch.randint(-8, 9, (Vd, r), generator=g).float() / 16).half()
    last = torch.randint(0, Vd, (B,), generator=g, dtype=torch.int32)
    d_logits, ids = logits.cuda(), torch.full((B * k,), -1, dtype=torch.int32, device="cuda")
    ws = torch.empty(hs.hspec_markov_workspace_bytes(B, Vd, r), dtype=torch.uint8, device="cuda")
    hs.hspec_op_markov_head(d_logits, W_in.cuda(), W_out.cuda(), last.cuda(), None, ids, B, k, write, ws)
    prev, want, adj = last.long().cuda(), [], []
    for i in range(k):
        row = logits.view(B, k, Vd)[:, i].cuda().double() + W_in.cuda()[prev].double() @ W_out.cuda().double().t()
        prev = torch.from_numpy(row.cpu().numpy().argmax(1)).cuda()          # numpy's arg-max takes the first of equal values
        want.append(prev)
        adj.append(row)
    assert torch.equal(ids.view(B, k).long(), torch.stack(want, 1))
    expect = torch.stack(adj, 1).view(B * k, Vd).float() if write else logits.cuda()
    assert torch.equal(d_logits, expect)
    assert hs.hspec_op_device_status()["rc"] == 0


# states of up to 16 values per channel: the kernel's register sizes (4, 16) and what they round up, head counts per group that give
# one, two and four heads per block, head widths that leave threads idle, blocks of positions around its chunk of eight
@pytest.mark.parametrize("B,k,H,P,N,G,d_conv", [(2, 1, 12, 64, 4, 1, 4), (3, 8, 12, 64, 4, 4, 4), (2, 9, 6, 24, 3, 2, 3), (1, 32, 5, 128, 16, 1, 4),
                                                (2, 17, 8, 10, 5, 1, 1), (2, 7, 4, 64, 1, 2, 2)])
@pytest.mark.parametrize("dt_given,state", [(True, True), (False, True), (False, False)])
def test_scan_with_a_small_state(hs, B, k, H, P, N, G, d_conv, dt_given, state):
    import numpy as np
    from oracle import hspec_oracle as O
    Di, d_xBC = H * P, H * P + 2 * G * N
    ld = Di + d_xBC + (0 if dt_given else H)
    f32 = torch.float32
    zx, dt_raw = _rand((B * k, ld), 1, f32), _rand((B * k, H), 2, f32) if dt_given else None
    s0 = _rand((B, H, P, N), 3, torch.float16, 1.5) if state else None
    conv_w, conv_b = _rand((d_xBC, d_conv), 4, f32, 0.3), _rand((d_xBC,), 5, f32, 0.02)
    A_log, dt_bias, D = _rand((H,), 6, f32).abs(), _rand((H,), 7, f32) - 4.0, 1 + _rand((H,), 8, f32, 0.1)
    y = torch.full((B * k, Di), float("nan"), device="cuda")
    hs.hspec_op_mamba_scan(zx, dt_raw, s0, conv_w, conv_b, dt_bias, A_log, D, y, B, k, Di, P, N, G, d_conv)
    f64 = lambda t: t.double().cpu().numpy()
    for b in range(B):
        rows = f64(zx)[b * k:(b + 1) * k]
        xBC = O.conv_silu(rows[:, Di:Di + d_xBC], f64(conv_w), f64(conv_b))
        dt, a = O.discretise(f64(dt_raw)[b * k:(b + 1) * k] if dt_given else rows[:, Di + d_xBC:], f64(dt_bias), f64(A_log))
        S = f64(s0)[b] if state else np.zeros((H, P, N))
        yy, _ = O.scan_sequential(S, xBC[:, :Di].reshape(k, H, P), xBC[:, Di:Di + G * N].reshape(k, G, N),
                                  xBC[:, Di + G * N:].reshape(k, G, N), dt, a, f64(D))
        ref = yy.reshape(k, Di) * O.silu(rows[:, :Di])
        got = f64(y)[b * k:(b + 1) * k]
        # fp32 arithmetic over at most 32 positions and 16 state values, SiLU with the fast exponential and division (a few ulp
        # each): 1e-5 of the output's RMS leaves an order of magnitude
        assert np.abs(got - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max()), np.abs(got - ref).max()


# the general kernel on both sides of its rule: 592 blocks (four to an SM), 629 and 740 of them (five), 777; and 629 with the shared memory
# (43.6 KB) of which just five fit an SM and that (45.9 KB) of which four do.  With 60 state values the tolerance still leaves a factor
# of four: sums of 60 fp32 products are off by at most 60 x 6e-8 of their terms' absolute sum, typically by the root of that.
@pytest.mark.parametrize("B,k,H,P,N,G,d_conv", [(16, 3, 37, 64, 17, 37, 4), (17, 32, 37, 10, 17, 1, 4), (20, 2, 37, 24, 20, 1, 4), (21, 1, 37, 24, 20, 1, 4),
                                                (17, 9, 37, 64, 60, 1, 3), (17, 4, 37, 128, 32, 1, 2)])
@pytest.mark.parametrize("dt_given,state", [(True, True), (False, False)])
def test_scan_with_many_blocks(hs, B, k, H, P, N, G, d_conv, dt_given, state):
    test_scan_with_a_small_state(hs, B, k, H, P, N, G, d_conv, dt_given, state)


# rows that take clusters of 8, 4, 2 and 1 blocks; vocabularies below the split, at its edges, not a multiple of four (scalar tail, and
# rows off the 16-byte boundary)
@pytest.mark.parametrize("M", [1, 37, 74, 148, 296])
@pytest.mark.parametrize("V", [1, 8191, 8192, 32768, 65535])
def test_token_probs_row_splits(hs, M, V):
    z = _rand((M, V), M + V, torch.float32, 3.0)
    z[:, V // 2] += 8.0
    z[0, 0] = float("-inf")
    if V > 1:
        z[M - 1, :V - 1] = float("-inf")                    # all of the mass in the last share
    ids = torch.randint(0, V, (M,), device="cuda", dtype=torch.int32)
    ids[M - 1] = V - 1
    p = torch.full((M,), float("nan"), device="cuda")
    hs.hspec_op_token_probs(z, ids, p)
    ref = torch.softmax(z.double(), 1).gather(1, ids.long()[:, None])[:, 0]
    if V == 1:
        ref[0] = float("nan")                               # a row of -inf only has no probabilities
    # exponentials to 2^-21 relative (argument below 2^5, two ulp), sums of positive terms
    assert torch.allclose(p.double(), ref, rtol=2e-5, atol=1e-30, equal_nan=True)


# the first layer's in-projection runs on B + 1 rows: one request, a block of one position (no shared row), a row count that crosses
# into the many-row kernel (257) while the block has more, low-rank dt
@pytest.mark.parametrize("B,k,over", [(1, 2, dict()), (3, 1, dict()), (256, 2, dict()), (4, 3, dict(dt_rank=16, N=16)), (2, 4, dict(N=32))])
def test_step_with_shared_first_layer_rows(hs, B, k, over):
    import synth
    from harness import check_step, cuda_setup
    cfg = synth.derived(dict(dict(D=256, n_fuse=1, r=256, L=2, has_attn=[1, 0], kv_slot=[0, -1], n_slots=1, Di=512, P=64, N=128, G=1,
                                  d_conv=4, dt_rank=0, Hq=4, Hkv=2, dh=64, rope_theta=1.0e4, window=0, qk_norm=1, F=512, V=600,
                                  rms_eps=1e-6, page_size=16, name="rows", B=B, k=k, ctx=("const", 20, 20)), **over))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[5 + (b % 30) for b in range(B)])
    check_step(cfg, drafter, w, batch, k, requests=sorted({0, B // 2, B - 1}), what=f"rows {B} {k} {over}")
    drafter.close()


# few rows: K-slices inside a cluster of 2 to 8 CTAs (slice counts that divide the k-steps and that do not, rows that leave some CTAs of
# the cluster without a column), at the row counts where the tile width and the kernel change (16, 32, 128, 129)
@pytest.mark.parametrize("M", [1, 7, 16, 17, 32, 33, 100, 128, 129, 255])
@pytest.mark.parametrize("n_out,K", [(256, 4096), (130, 1000), (4096, 2048), (9000, 520), (17000, 640)])
@pytest.mark.parametrize("kind", ["f32", "accumulate", "f16"])
def test_few_row_gemm_slices(hs, M, n_out, K, kind):
    _gemm_against_fp64(hs, M, n_out, K, kind)


def _attention_against_fp64(hs, ctx, k, rep, window, chunk, dh, Hkv, page=16):
    import numpy as np
    B, Hq = len(ctx), Hkv * rep
    pages = [(c + page - 1) // page for c in ctx]
    perm = torch.randperm(sum(pages), generator=torch.Generator().manual_seed(3)).int()
    table, at = torch.full((B, max(pages)), -1, dtype=torch.int32), 0
    for b, n in enumerate(pages):
        table[b, :n] = perm[at:at + n]
        at += n
    bf = torch.bfloat16
    kp, vp = _rand((sum(pages), page, Hkv, dh), 1, bf), _rand((sum(pages), page, Hkv, dh), 2, bf)
    q, kb, vb = _rand((B * k, Hq, dh), 4, bf), _rand((B * k, Hkv, dh), 5, bf), _rand((B * k, Hkv, dh), 6, bf)
    o = torch.full((B * k, Hq * dh), float("nan"), dtype=torch.float16, device="cuda")
    ws = torch.empty(hs.hspec_attention_workspace_bytes(B, k, Hq, Hkv, dh, max(ctx), window, chunk), dtype=torch.uint8, device="cuda")
    table, lens = table.cuda(), torch.tensor(ctx, dtype=torch.int32).cuda()
    for _ in range(3):            # a work list read before it is written is an empty one here, and leaves NaN
        ws.zero_()
        o.fill_(float("nan"))
        hs.hspec_op_attention(q, kb, vb, kp, vp, table, lens, max(ctx), o, B, k, Hq, Hkv, dh, page, window, chunk, ws)
        assert not bool(o.isnan().any())
    for b, c in enumerate(ctx):
        rows = table[b, :pages[b]].long()
        K = torch.cat([kp[rows].reshape(-1, Hkv, dh)[:c], kb[b * k:(b + 1) * k]]).double()
        V = torch.cat([vp[rows].reshape(-1, Hkv, dh)[:c], vb[b * k:(b + 1) * k]]).double()
        pos_q, pos_k = torch.arange(c, c + k, device="cuda"), torch.arange(c + k, device="cuda")
        d = pos_q[:, None] - pos_k[None, :]
        vis = (d >= 0) & ((d < window) if window else torch.ones_like(d, dtype=torch.bool))
        s = torch.einsum("ihrd,jhd->ihrj", q[b * k:(b + 1) * k].view(k, Hkv, rep, dh).double(), K) / np.sqrt(dh)
        p = torch.softmax(s.masked_fill(~vis[:, None, None, :], float("-inf")), -1)
        ref = torch.einsum("ihrj,jhd->ihrd", p, V).reshape(k, Hq * dh)
        # softmax weights enter the product as bf16 (2^-9 relative each), the rest is fp32, the result fp16 (2^-11): relative to the sum of
        # |weight x value|, with a factor 2 for the exponentials
        mag = torch.einsum("ihrj,jhd->ihrd", p, V.abs()).reshape(k, Hq * dh)
        err = (o[b * k:(b + 1) * k].double() - ref).abs()
        assert bool((err <= 2.0 ** -8 * mag + 2.0 ** -11 * ref.abs() + 1e-6).all()), float((err / mag).max())


# query rows per KV head at the edges of the row copies (4 copies up to 32 rows, 2 up to 64, 1 above), contexts that end inside a copy's
# part of a tile, a block that starts a tile of its own, single and several chunks, the window's leading edge inside a part; head width
# 64: the other kernel, four and two warps per 16 rows, and one above 64 rows
@pytest.mark.parametrize("k,rep", [(1, 1), (8, 4), (11, 3), (32, 1), (16, 4), (32, 2), (13, 5), (16, 8)])
@pytest.mark.parametrize("window,chunk", [(0, 0), (0, 256), (300, 0), (0, 64)])
@pytest.mark.parametrize("dh,Hkv", [(128, 2), (64, 2), (64, 8)])
def test_attention_row_copies(hs, k, rep, window, chunk, dh, Hkv):
    _attention_against_fp64(hs, [0, 1, 31, 97, 128, 500, 1111], k, rep, window, chunk, dh, Hkv)


# the mma.sync kernel's forms: four, two and one warps per 16 query rows, on either side of the CTA counts that choose between them (8 KV heads,
# one chunk: 37 | 38 requests with heads of 64, 18 | 19 with heads of 128); heads of 128 come here with pages that are not 16 tokens
@pytest.mark.parametrize("dh,page,B,Hkv,k,rep", [(64, 16, 75, 8, 1, 1), (64, 16, 37, 8, 8, 4), (64, 16, 38, 8, 8, 4), (64, 16, 37, 8, 12, 4), (64, 16, 38, 8, 12, 4),
                                                 (64, 16, 18, 8, 16, 4), (64, 16, 38, 8, 16, 4), (128, 32, 3, 2, 4, 4), (128, 8, 18, 8, 8, 4),
                                                 (128, 128, 19, 8, 8, 4), (128, 8, 75, 8, 12, 4), (128, 8, 18, 8, 16, 4), (128, 64, 19, 8, 16, 4),
                                                 (128, 5, 2, 2, 16, 8), (128, 1, 1, 1, 32, 16)])
@pytest.mark.parametrize("window", [0, 40])
def test_attention_warps_per_row(hs, dh, page, B, Hkv, k, rep, window):
    _attention_against_fp64(hs, [(37 * b + 61) % 129 for b in range(B)], k, rep, window, 256, dh, Hkv, page)


# the norm behind a residual GEMM adds the GEMM's K-sliced tail tiles: two slices and three to eight (behind the out and the down projection, as asserted),
# one (nothing to add), all tail and a whole wave in front of it; widths that take 256 and 512 threads and those that no longer fit the norm's
# registers (6 x 4 x 256 and 6 x 4 x 512 floats); hidden state asked for
@pytest.mark.parametrize("D,F,B,k,out_slices,down_slices", [(512, 4096, 9, 32, 2, 8), (4096, 2048, 20, 13, 1, 1), (4096, 4096, 5, 29, 1, 4), (2048, 4096, 9, 31, 1, 4),
                                                          (7168, 1024, 9, 30, 1, 1), (12544, 512, 10, 26, 1, 1), (12544, 4096, 10, 26, 1, 3), (12800, 4096, 9, 31, 1, 2),
                                                          (1280, 1024, 141, 32, 1, 1)])
def test_residual_tail_is_added_by_the_norm(hs, D, F, B, k, out_slices, down_slices):
    assert (hs.hspec_debug_gemm_tiles(B * k, D, 1024)[1], hs.hspec_debug_gemm_tiles(B * k, D, F)[1]) == (out_slices, down_slices)
    import synth
    from harness import check_step, cuda_setup
    cfg = synth.derived(dict(D=D, n_fuse=1, r=64, L=1, has_attn=[0], kv_slot=[-1], n_slots=0, Di=1024, P=64, N=4, G=1, d_conv=4, dt_rank=0,
                             Hq=2, Hkv=1, dh=64, rope_theta=1.0e4, window=0, qk_norm=1, F=F, V=300, rms_eps=1e-6, page_size=16, name="tail",
                             B=B, k=k, ctx=("const", 16, 16)))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[16] * B)
    check_step(cfg, drafter, w, batch, k, requests=[0, B - 1], what=f"tail {D} {F}")
    drafter.close()

# small states: the gated norm runs in the scan's own kernel as long as a request's blocks fit a cluster of eight (here one to eight blocks,
# head counts per group that are no power of two, and one too many: 9 blocks), low-rank dt up to the width where a GEMM expands it instead
@pytest.mark.parametrize("Di,P,N,G,dt_rank,B,k", [(256, 64, 16, 1, 16, 1, 1), (3072, 64, 4, 4, 0, 3, 8), (1152, 64, 4, 9, 0, 2, 5), (2048, 64, 16, 8, 64, 2, 32),
                                                  (2304, 64, 3, 36, 0, 2, 4), (640, 32, 8, 5, 40, 3, 9), (512, 64, 16, 2, 72, 2, 3), (960, 120, 4, 1, 8, 2, 17)])
def test_small_state_scan_with_norm(hs, Di, P, N, G, dt_rank, B, k):
    import synth
    from harness import check_step, cuda_setup
    cfg = synth.derived(dict(D=256, n_fuse=1, r=64, L=2, has_attn=[0, 0], kv_slot=[-1, -1], n_slots=0, Di=Di, P=P, N=N, G=G, d_conv=4, dt_rank=dt_rank,
                             Hq=4, Hkv=2, dh=64, rope_theta=1.0e4, window=0, qk_norm=1, F=512, V=600, rms_eps=1e-6, page_size=16, name="small",
                             B=B, k=k, ctx=("const", 20, 20)))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[20] * B)
    check_step(cfg, drafter, w, batch, k, requests=list(range(B)), what=f"small {Di} {P} {N} {G} {dt_rank}")
    drafter.close()


# the QK norm behind the QKV projection adds that GEMM's K-sliced tail tiles up to 512 rows (513 and a whole wave with a tail behind it take the pass
# of their own, where there are slices): one slice to eight, as asserted; heads of a quarter and of half a weight tile, a last weight tile that is only part full
@pytest.mark.parametrize("D,dh,Hq,Hkv,B,k,slices", [(1024, 64, 16, 4, 9, 32, 1), (1024, 128, 8, 2, 9, 32, 1), (1024, 128, 6, 1, 20, 13, 1), (1024, 128, 8, 2, 16, 32, 1),
                                                     (1024, 64, 14, 2, 27, 19, 1), (1024, 64, 14, 2, 141, 32, 1), (1024, 64, 14, 2, 5, 29, 2), (2048, 64, 16, 4, 9, 32, 4),
                                                     (2048, 128, 6, 1, 20, 13, 4), (2048, 128, 8, 2, 16, 32, 3), (2048, 64, 14, 2, 27, 19, 4), (4096, 128, 8, 2, 9, 32, 6),
                                                     (4096, 64, 14, 2, 5, 29, 7)])
def test_qkv_tail_is_added_by_the_qk_norm(hs, D, dh, Hq, Hkv, B, k, slices):
    import synth
    from harness import check_step, cuda_setup
    assert hs.hspec_debug_gemm_tiles(B * k, (Hq + 2 * Hkv) * dh, D)[1] == slices
    cfg = synth.derived(dict(D=D, n_fuse=1, r=64, L=1, has_attn=[1], kv_slot=[0], n_slots=1, Di=1024, P=64, N=4, G=1, d_conv=4, dt_rank=0,
                             Hq=Hq, Hkv=Hkv, dh=dh, rope_theta=1.0e4, window=0, qk_norm=1, F=512, V=600, rms_eps=1e-6, page_size=16, name="qkvtail",
                             B=B, k=k, ctx=("const", 20, 20)))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[b % 40 for b in range(B)])
    check_step(cfg, drafter, w, batch, k, requests=sorted({0, 1, B // 2, B - 1}), what=f"qkv tail {dh} {B}")
    drafter.close()


# the arg-max across tiles: equal values in one tile, in neighbouring and in distant ones (lowest index wins), +0 against -0, rows of negative
# values only; one-CTA kernel and pair kernel, one activation tile and several, a single vocabulary row
@pytest.mark.parametrize("M", [1, 9, 128, 129, 600])
@pytest.mark.parametrize("V", [1, 127, 300, 20000])
@pytest.mark.parametrize("alloc", [True, False])
def test_lm_head_argmax_ties(hs, M, V, alloc):
    K = 64
    if not alloc and M > 512:
        pytest.skip("more rows than the built-in scratch takes")
    x, W = _rand((M, K), 1, torch.float16), _rand((V, K), 2, torch.float16)
    W[V // 2] = W[0]                                          # a tie far away
    W[min(V - 1, 3)] = W[0]
    x[M // 2] = -x[M // 2].abs()
    x[0] = 0.                                                 # every logit is +0 or -0: index 0
    ids = torch.full((M,), -1, dtype=torch.int32, device="cuda")
    logits = torch.empty((M, V), device="cuda")
    for _ in range(2):                                        # the second call starts from what the first one left
        ids.fill_(-1)
        if alloc:
            ws = torch.full((((V + 127) // 128) * M * 8 + 1024,), 255, dtype=torch.uint8, device="cuda")
            hs.hspec_op_lm_head_argmax(x, W, ids, logits, ws)
        else:
            hs.hspec_op_lm_head_argmax_noalloc(x, W, ids, logits=logits)
        z = logits.clone()
        best = z.max(1, keepdim=True).values
        first = torch.where(z == best, torch.arange(V, device="cuda"), V).min(1).values.int()     # exact: the kernel's own logits
        assert torch.equal(ids, first)


# logits that rise along the vocabulary (every column group reaches its rows' maxima so far and runs the reduction), that fall (only the first ones do) and
# that are all the same; whole and part tiles, with logits written and without
@pytest.mark.parametrize("M", [33, 77, 128, 300])
@pytest.mark.parametrize("V", [16384, 16500, 40001])
@pytest.mark.parametrize("write", [True, False])
def test_lm_head_argmax_in_its_worst_orders(hs, M, V, write):
    K, v = 64, torch.arange(V, device="cuda")
    x, W = torch.zeros((M, K), dtype=torch.float16, device="cuda"), _rand((V, K), 2, torch.float16)
    W[:, 0], W[:, 1] = (v // 128 * 128).half(), (v % 128).half()                  # v, exactly, over two columns
    x[0::3, :2], x[1::3, :2] = 1.0, -1.0
    want = torch.zeros(M, dtype=torch.int32, device="cuda")
    want[0::3] = V - 1
    ids, logits = torch.full((M,), -1, dtype=torch.int32, device="cuda"), torch.full((M, V), float("nan"), device="cuda") if write else None
    hs.hspec_op_lm_head_argmax_noalloc(x, W, ids, logits=logits)
    assert torch.equal(ids, want)
    ws = torch.full((((V + 127) // 128) * M * 8 + 1024,), 255, dtype=torch.uint8, device="cuda")
    hs.hspec_op_lm_head_argmax(x, W, ids.fill_(-1), logits, ws)
    assert torch.equal(ids, want)
    if write:
        assert torch.equal(logits[0], v.float()) and torch.equal(logits[1], -v.float()) and not bool(logits[2].any())


# a NaN logit counts as -inf: one at the first and the last row of a tile and of the matrix, next to and away from the maximum, a row that is
# all NaN (index 0), +inf (chosen), -inf; one-CTA kernel and pair kernel, a last tile that is part full
@pytest.mark.parametrize("M", [5, 40, 200])
@pytest.mark.parametrize("V", [130, 300, 20000])
def test_lm_head_argmax_takes_nan_as_minus_infinity(hs, M, V):
    K = 64
    x, W = _rand((M, K), 1, torch.float16), _rand((V, K), 2, torch.float16)
    x[:, 0] = 1.0
    x[1, 0] = -1.0
    x[2] = float("nan")
    nan, inf = float("nan"), float("inf")
    for v in {0, 31, 32, 127, 128, V // 2, V - 1}:
        W[v, 1] = nan
    ids = torch.empty(M, dtype=torch.int32, device="cuda")
    logits = torch.empty((M, V), device="cuda")
    ws = torch.empty(((V + 127) // 128) * M * 8 + 1024, dtype=torch.uint8, device="cuda")
    for big in (None, 5, V - 2):                              # (+inf in every row but row 1, where it is -inf)
        if big is not None:
            W[big, 0] = inf
        ids.fill_(-1)
        hs.hspec_op_lm_head_argmax(x, W, ids, logits, ws)
        z = logits.nan_to_num(nan=-inf, posinf=inf, neginf=-inf)
        first = torch.where(z == z.max(1, keepdim=True).values, torch.arange(V, device="cuda"), V).min(1).values.int()
        assert bool(logits[2].isnan().all()) and bool((logits[0].isnan().sum() >= 6).item())
        assert torch.equal(ids, first) and int(ids[2]) == 0
        hs.hspec_op_lm_head_argmax_noalloc(x, W, ids.fill_(-1), logits=logits)
        assert torch.equal(ids, first)


# the same for the causal-correction head, in one launch (up to 128 requests) and position by position, with and without a pruned vocabulary
@pytest.mark.parametrize("B", [3, 100, 131])
@pytest.mark.parametrize("pruned", [False, True])
def test_markov_head_takes_nan_as_minus_infinity(hs, B, pruned):
    k, Vd, r, V = 4, 19300, 64, 25000
    g = torch.Generator().manual_seed(B)
    logits = (torch.randint(-256, 257, (B, k, Vd), generator=g).float() / 64).cuda()
    nan, inf = float("nan"), float("inf")
    logits[:, :, [0, 31, 32, 128, Vd // 2, Vd - 1]] = nan
    logits[0, 1] = nan                                        # row 0, and the next position goes on from it
    logits[1, 0] = -inf
    logits[1, 2, 700] = inf
    logits[2, 3, 500] = -inf
    W_in = (torch.randint(-8, 9, (V, r), generator=g).float() / 16).half().cuda()
    W_out = (torch.randint(-8, 9, (Vd, r), generator=g).float() / 16).half().cuda()
    id_map = torch.sort(torch.randperm(V, generator=g)[:Vd])[0].int().cuda() if pruned else None
    last = torch.randint(0, V, (B,), generator=g, dtype=torch.int32).cuda()
    ids = torch.full((B * k,), -1, dtype=torch.int32, device="cuda")
    out = logits.clone().view(B * k, Vd)
    ws = torch.empty(hs.hspec_markov_workspace_bytes(B, Vd, r), dtype=torch.uint8, device="cuda")
    hs.hspec_op_markov_head(out, W_in, W_out, last, id_map, ids, B, k, True, ws)
    prev = last.long()
    for i in range(k):                                        # (exact in fp32, as in the test above)
        row = logits[:, i].double() + W_in[prev].double() @ W_out.double().t()
        assert torch.equal(out.view(B, k, Vd)[:, i].nan_to_num(nan=777.0), row.float().nan_to_num(nan=777.0))
        row = row.nan_to_num(nan=-inf, posinf=inf, neginf=-inf)
        best = torch.where(row == row.max(1, keepdim=True).values, torch.arange(Vd, device="cuda"), Vd).min(1).values
        prev = id_map[best].long() if pruned else best
        assert torch.equal(ids.view(B, k)[:, i].long(), prev), i
    assert hs.hspec_op_device_status()["rc"] == 0


def test_markov_head_where_cooperative_launches_are_refused():
    """The tests of the one-launch form again, in a process in which that launch is refused: same ids, same logits, position by position."""
    import os
    import subprocess
    import sys
    res = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", __file__, "-k",
                          "test_markov_head_chunks_and_tiles or test_markov_head_takes_nan"],
                         env=dict(os.environ, HSPEC_NO_COOPERATIVE="1"), capture_output=True, text=True, timeout=300,
                         cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert res.returncode == 0 and " passed" in res.stdout, res.stdout[-3000:] + res.stderr[-1000:]


# low-rank dt that the scan expands itself, at the states the other scan kernels take: the stream kernel (N = 128, one and two tiles of 16
# positions), the generic one (N = 32), on either side of the product count (2^22) and of the rank (64) above which a GEMM does it; bf16 operands
@pytest.mark.parametrize("Di,N,G,dt_rank,B,k,bf16", [(512, 128, 1, 16, 2, 16, 0), (512, 128, 2, 64, 3, 17, 0), (512, 128, 2, 64, 3, 32, 1), (512, 128, 1, 72, 2, 5, 0),
                                                     (768, 32, 1, 16, 2, 9, 0), (768, 32, 3, 64, 2, 32, 0), (4096, 128, 4, 64, 32, 32, 0), (4096, 128, 4, 64, 33, 32, 0)])
def test_low_rank_dt_in_the_scan(hs, Di, N, G, dt_rank, B, k, bf16):
    import synth
    from harness import check_step, cuda_setup
    cfg = synth.derived(dict(D=256, n_fuse=1, r=64, L=2, has_attn=[0, 0], kv_slot=[-1, -1], n_slots=0, Di=Di, P=64, N=N, G=G, d_conv=4, dt_rank=dt_rank,
                             Hq=4, Hkv=2, dh=64, rope_theta=1.0e4, window=0, qk_norm=1, F=512, V=600, rms_eps=1e-6, page_size=16, name="lowrank",
                             act_bf16=bf16, B=B, k=k, ctx=("const", 20, 20)))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[20] * B)
    check_step(cfg, drafter, w, batch, k, requests=[0, B - 1], what=f"low rank {Di} {N} {dt_rank} {B}", **(dict(tol=5e-2) if bf16 else {}))
    drafter.close()


# the scan of the serving shapes (P = 64, N = 128), with scratch: one tile of 16 positions and two, on both sides; few blocks and several waves of
# them; groups of four heads and one group of all; rows of 16-byte multiples (vector loads of the conv), of 8-byte ones (scalar) and, off the 8 bytes,
# the general kernel; no state
@pytest.mark.parametrize("B,k,H,G,ld_extra,state,d_conv", [(1, 1, 4, 1, 0, True, 4), (3, 15, 8, 2, 0, True, 4), (41, 16, 64, 16, 0, True, 4), (41, 17, 64, 16, 0, True, 4),
                                                           (75, 32, 32, 1, 0, True, 4), (40, 9, 36, 3, 1, True, 4), (40, 31, 36, 3, 2, True, 4), (64, 5, 32, 2, 0, False, 4),
                                                           (2, 9, 8, 2, 0, True, 3), (2, 17, 8, 2, 0, True, 2), (2, 32, 8, 2, 2, True, 1)])
def test_scan_tiles_on_tensor_cores(hs, B, k, H, G, ld_extra, state, d_conv):
    import numpy as np
    from oracle import hspec_oracle as O
    P, N = 64, 128
    Di, d_xBC, f32 = H * P, H * P + 2 * G * N, torch.float32
    ld = Di + d_xBC + H + ld_extra
    zx = _rand((B * k, ld), 1, f32)
    s0 = _rand((B, H, P, N), 3, torch.float16, 1.5) if state else None
    conv_w, conv_b = _rand((d_xBC, d_conv), 4, f32, 0.3), _rand((d_xBC,), 5, f32, 0.02)
    A_log, dt_bias, D = _rand((H,), 6, f32).abs(), _rand((H,), 7, f32) - 4.0, 1 + _rand((H,), 8, f32, 0.1)
    y = torch.full((B * k, Di), float("nan"), device="cuda")
    ws = torch.full((hs.hspec_scan_workspace_bytes(B, k, Di, N, G),), 255, dtype=torch.uint8, device="cuda")      # NaN wherever nothing is written
    hs.hspec_op_mamba_scan(zx, None, s0, conv_w, conv_b, dt_bias, A_log, D, y, B, k, Di, P, N, G, d_conv, ws)
    assert bool(torch.isfinite(y).all())
    f64 = lambda t: t.double().cpu().numpy()
    for b in sorted({0, 1 % B, B // 2, B - 1}):
        rows = f64(zx[b * k:(b + 1) * k])
        xBC = O.conv_silu(rows[:, Di:Di + d_xBC], f64(conv_w), f64(conv_b))
        dt, a = O.discretise(rows[:, Di + d_xBC:Di + d_xBC + H], f64(dt_bias), f64(A_log))
        S = f64(s0[b]) if state else np.zeros((H, P, N))
        yy, _ = O.scan_sequential(S, xBC[:, :Di].reshape(k, H, P), xBC[:, Di:Di + G * N].reshape(k, G, N),
                                  xBC[:, Di + G * N:].reshape(k, G, N), dt, a, f64(D))
        ref = yy.reshape(k, Di) * O.silu(rows[:, :Di])
        got = f64(y[b * k:(b + 1) * k])
        # sums of 128 products with C in 22 bits and of up to 32 with both factors in 21 or 22; exp(x), in SiLU and decay, to about (2 + |x|) x 2^-23 of itself
        # (x log2 e is rounded before the power), so of no weight where |x| is large and the value e^-|x|: in all some 3 x 2^-22 of the
        # result, RMS over RMS (4.9e-7 to 6e-7 measured; twice that allowed), and at a single place 10 x 2^-22 of the terms' absolute sum, which is below 20 RMS
        assert np.sqrt(((got - ref) ** 2).mean()) <= 6 * 2.0 ** -22 * np.sqrt((ref ** 2).mean())
        assert np.abs(got - ref).max() <= 1e-4 * max(1.0, np.sqrt((ref ** 2).mean())), np.abs(got - ref).max()
    assert hs.hspec_op_device_status()["rc"] == 0


# Draws on a grid, from integers alone: the same bits on every platform.
def _grid(shape, seed, low, high, dtype=torch.float32):
    import numpy as np
    v = np.random.default_rng(seed).integers(0, 1 << 16, size=shape)
    return torch.from_numpy((low + (high - low) * v / 65536.0).astype(np.float32)).to("cuda", dtype)


def _scan_of_few_rows(hs, B, k, H, G, state, a_log=(0.0, 2.0), scratch=True):
    P, N = 64, 128
    Di, d_xBC = H * P, H * P + 2 * G * N
    zx = _grid((B * k, Di + d_xBC + H), 1, -2.0, 2.0)
    s0 = _grid((B, H, P, N), 2, -2.0, 2.0, torch.float16) if state else None
    conv_w, conv_b = _grid((d_xBC, 4), 3, -0.5, 0.5), _grid((d_xBC,), 4, -0.05, 0.05)
    dt_bias, A_log, D = _grid((H,), 5, -6.0, -2.0), _grid((H,), 6, *a_log), _grid((H,), 7, 0.5, 1.5)
    y = torch.full((B * k, Di), float("nan"), device="cuda")
    ws = torch.full((hs.hspec_scan_workspace_bytes(B, k, Di, N, G),), 255, dtype=torch.uint8, device="cuda") if scratch else None
    hs.hspec_op_mamba_scan(zx, None, s0, conv_w, conv_b, dt_bias, A_log, D, y, B, k, Di, P, N, G, 4, ws)
    return y


# A step's logits carry the scan's last bits through the 16-bit roundings behind it, up to 5e-4 (fp16 operands) and 4e-3 (bf16) of their size, and
# there the arg-max of near-tied tokens turns: of a few tokens, one is several per cent.  So the sums of this path keep their order, and its
# outputs are compared to the bit with those on record (CRC-32 of the fp32 outputs).
@pytest.mark.parametrize("B,k,H,G,state", [(1, 1, 4, 1, True), (1, 16, 128, 4, True), (1, 17, 128, 4, True), (2, 32, 8, 2, True), (3, 29, 64, 4, True),
                                           (5, 7, 128, 4, True), (3, 16, 64, 4, False), (8, 20, 16, 1, False)])
def test_scan_outputs_keep_their_bits(hs, B, k, H, G, state):
    import json
    import os
    import zlib
    y = _scan_of_few_rows(hs, B, k, H, G, state)
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "scan_crc32.json")) as f:
        want = json.load(f)
    assert zlib.crc32(y.cpu().numpy().tobytes()) == want["%d,%d,%d,%d,%d" % (B, k, H, G, state)]


# Prefix sums of dt A at -infinity: exp of their differences is NaN, with scratch as without, and is not turned into a factor.
def test_scan_lets_a_nan_decay_through(hs):
    with_scratch = _scan_of_few_rows(hs, 2, 9, 8, 2, True, a_log=(100.0, 101.0))
    without = _scan_of_few_rows(hs, 2, 9, 8, 2, True, a_log=(100.0, 101.0), scratch=False)
    assert bool(torch.isnan(without).all()) and bool(torch.isnan(with_scratch).all())


# The scan allocates nothing, also as the first call of a process: it can be captured.
def test_scan_as_a_process_first_call_under_capture():
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import torch, paper_2609_24197_b200 as hs; hs.load_library()\n"
            "B, k, H, P, N, G = 2, 5, 8, 64, 128, 2; Di = H * P; W = Di + 2 * G * N\n"
            "r = lambda *s: torch.rand(s, device='cuda') - 0.5\n"
            "a = [r(B * k, Di + W + H), None, r(B, H, P, N).half(), r(W, 4), r(W), r(H), r(H), r(H)]; y = torch.zeros(B * k, Di, device='cuda')\n"
            "ws = torch.zeros(hs.hspec_scan_workspace_bytes(B, k, Di, N, G), dtype=torch.uint8, device='cuda')\n"
            "run = lambda: hs.hspec_op_mamba_scan(*a, y, B, k, Di, P, N, G, 4, ws)\n"
            "g = torch.cuda.CUDAGraph(); torch.cuda.synchronize()\n"
            "with torch.cuda.graph(g): run()\n"
            "g.replay(); torch.cuda.synchronize(); got = y.clone(); y.zero_(); run(); torch.cuda.synchronize()\n"
            "assert bool(got.any()) and torch.equal(got, y); print('same')\n")
    res = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and "same" in res.stdout, res.stdout[-2000:] + res.stderr[-2000:]


# Operands off the boundaries that the vector loads of a path want: state (16-bit values) 2, 8 and 16 bytes behind a 32-byte boundary, rows in and out
# 4 and 8 bytes behind a 16-byte one, scratch 8; the serving shapes and the general kernel, with scratch and without.  Each call has to give what the
# aligned one gives: two kernels' fp32 sums of 128 products (2^-22 of some 20 RMS, as above).
@pytest.mark.parametrize("P,N", [(64, 128), (24, 40)])
@pytest.mark.parametrize("off_state,off_in,off_out,off_ws", [(1, 0, 0, 0), (4, 0, 0, 0), (8, 0, 0, 0), (0, 1, 0, 0), (0, 2, 0, 0), (0, 0, 1, 0), (0, 0, 2, 0), (0, 0, 0, 8),
                                                             (4, 1, 1, 8)])
@pytest.mark.parametrize("scratch", [True, False])
def test_scan_of_misaligned_operands(hs, P, N, off_state, off_in, off_out, off_ws, scratch):
    B, k, H, G, f32 = 2, 18, 8, 2, torch.float32
    Di, d_xBC = H * P, H * P + 2 * G * N
    conv_w, conv_b = _rand((d_xBC, 4), 4, f32, 0.3), _rand((d_xBC,), 5, f32, 0.02)
    A_log, dt_bias, D = _rand((H,), 6, f32).abs(), _rand((H,), 7, f32) - 4.0, 1 + _rand((H,), 8, f32, 0.1)
    zx, s0 = _rand((B * k, Di + d_xBC + H), 1, f32), _rand((B, H, P, N), 3, torch.float16, 1.5)

    def at(t, off):                                            # a copy of t, `off` elements into its storage
        flat = torch.empty(t.numel() + off, dtype=t.dtype, device="cuda")
        flat[off:] = t.flatten()
        return flat[off:].view(t.shape)

    def run(o_state, o_in, o_out, o_ws):
        y = at(torch.full((B * k, Di), float("nan"), device="cuda"), o_out)
        ws = at(torch.zeros(hs.hspec_scan_workspace_bytes(B, k, Di, N, G), dtype=torch.uint8, device="cuda"), o_ws) if scratch else None
        hs.hspec_op_mamba_scan(at(zx, o_in), None, at(s0, o_state), conv_w, conv_b, dt_bias, A_log, D, y, B, k, Di, P, N, G, 4, ws)
        return y
    want, got = run(0, 0, 0, 0), run(off_state, off_in, off_out, off_ws)
    assert float((got - want).abs().max()) <= 1e-4 * max(1.0, float(want.square().mean().sqrt()))


# the norm of wide rows, where a CTA fetches its next row ahead: one row per CTA and several, row lengths around 6144 (256 or 512 threads) and
# 12 288 (the row no longer fits the registers), one that is no multiple of four
@pytest.mark.parametrize("M", [1, 296, 297, 593])
@pytest.mark.parametrize("n", [6144, 6148, 8192, 12288, 12292, 7001])
def test_rmsnorm_rows_ahead(hs, M, n):
    x, w = _rand((M, n), 1, torch.float32, 3.0), 1 + _rand((n,), 2, torch.float32, 0.1)
    y = torch.full((M, n), float("nan"), dtype=torch.float16, device="cuda")
    before = x.clone()
    hs.hspec_op_rmsnorm(x, w, y, 1e-6)
    ref = x.double() / torch.sqrt((x.double() ** 2).mean(1, keepdim=True) + 1e-6) * w.double()
    # one fp16 rounding (2^-11 of the value) and a few fp32 ones
    assert bool(((y.double() - ref).abs() <= ref.abs() * 2.0 ** -10.9 + 1e-6).all())
    assert torch.equal(x, before)


# the norm of operands off the boundaries of its vector loads and stores (x and w 16 bytes, y 8), in one CTA per row and with rows ahead
@pytest.mark.parametrize("M,n", [(3, 256), (300, 8192)])
@pytest.mark.parametrize("off_x,off_w,off_y", [(1, 0, 0), (2, 0, 0), (0, 1, 0), (0, 0, 1), (0, 0, 4), (3, 2, 6)])
def test_rmsnorm_of_misaligned_operands(hs, M, n, off_x, off_w, off_y):
    x = _rand((M * n + off_x,), 1, torch.float32, 3.0)[off_x:].view(M, n)
    w = (1 + _rand((n + off_w,), 2, torch.float32, 0.1))[off_w:]
    y = torch.full((M * n + off_y,), float("nan"), dtype=torch.float16, device="cuda")[off_y:].view(M, n)
    hs.hspec_op_rmsnorm(x, w, y, 1e-6)
    ref = x.double() / torch.sqrt((x.double() ** 2).mean(1, keepdim=True) + 1e-6) * w.double()
    assert bool(((y.double() - ref).abs() <= ref.abs() * 2.0 ** -10.9 + 1e-6).all())


# Launches of the pair GEMM that take no K-slices add a row's products in the order of K, whatever the tile's width: a call's rows are the bits that the
# same rows have among others.  (Tiles of more than 256 rows, sliced where the others are not, moved the sums of 257 rows of 5120 and of 549 of 4096.)
@pytest.mark.parametrize("M,others,n_out,K", [(257, 300, 5120, 8192), (549, 640, 4096, 14336), (320, 301, 5120, 25600), (400, 512, 17536, 256)])
@pytest.mark.parametrize("kind", [torch.float16, torch.bfloat16])
def test_gemm_rows_keep_their_bits_among_others(hs, M, others, n_out, K, kind):
    x, W = _rand((max(M, others), K), 1, kind), _rand((n_out, K), 2, kind, 0.05)

    def rows(m):
        y = torch.full((m, n_out), float("nan"), device="cuda")
        hs.hspec_op_gemm(x[:m].contiguous(), W, y, workspace=torch.empty(hs.hspec_gemm_workspace_bytes(m, n_out, K), dtype=torch.uint8, device="cuda"))
        return y[:min(M, others)]
    assert torch.equal(rows(M), rows(others))


# the pair GEMM at 257 to 549 rows, where the rows are spread over two to four tiles: a whole wave and a tail of almost one, a last weight tile that is part full,
# K that ends in a part k-step or is shorter than one, one slice (most), two (270 rows) and three (257 of 2560)
@pytest.mark.parametrize("M,n_out,K", [(257, 17000, 520), (288, 17000, 512), (289, 17000, 72), (352, 17000, 128), (353, 17000, 192), (416, 17000, 64), (417, 17000, 512),
                                       (480, 17000, 512), (481, 17000, 8), (512, 17408, 256), (257, 5000, 4096), (270, 4096, 4096), (257, 2560, 4096),
                                       (549, 4096, 8192)])
@pytest.mark.parametrize("kind,out", [(torch.float16, torch.float32), (torch.float16, torch.float16), (torch.bfloat16, torch.bfloat16), (torch.float16, "add")])
def test_gemm_rows_over_several_tiles(hs, M, n_out, K, kind, out):
    x, W = _rand((M, K), 1, kind), _rand((n_out, K), 2, kind, 0.05)
    add = out == "add"
    y = _rand((M, n_out), 3, torch.float32) if add else torch.full((M, n_out), float("nan"), dtype=out, device="cuda")
    ref = x.double() @ W.double().t() + (y.double() if add else 0.)
    # every partial sum of K products is rounded to fp32 (2^-24): K / 64 roundings per element in a chain at most, here taken as 64; and the store's
    # rounding
    terms = x.double().abs() @ W.double().abs().t() + (y.double().abs() if add else 0.)
    store = {torch.float16: 2.0 ** -11, torch.bfloat16: 2.0 ** -8}.get(out, 2.0 ** -23)
    ws = torch.full((hs.hspec_gemm_workspace_bytes(M, n_out, K),), 255, dtype=torch.uint8, device="cuda")
    hs.hspec_op_gemm(x, W, y, accumulate=add, workspace=ws)
    assert bool(((y.double() - ref).abs() <= terms * 2.0 ** -18 + ref.abs() * store + 1e-7).all())
    assert hs.hspec_op_device_status()["rc"] == 0


# the SwiGLU epilogue with several tiles of rows: 300 and 512 rows
@pytest.mark.parametrize("B,k", [(30, 10), (16, 32)])
def test_gemm_rows_over_several_tiles_with_swiglu(hs, B, k):
    import synth
    from harness import check_step, cuda_setup
    cfg = synth.derived(dict(D=256, n_fuse=1, r=64, L=1, has_attn=[0], kv_slot=[-1], n_slots=0, Di=512, P=64, N=4, G=1, d_conv=4, dt_rank=0,
                             Hq=2, Hkv=1, dh=64, rope_theta=1.0e4, window=0, qk_norm=1, F=8512, V=300, rms_eps=1e-6, page_size=16, name="wide",
                             B=B, k=k, ctx=("const", 16, 16)))
    drafter, w, batch = cuda_setup(cfg, ctx_lens=[16] * B)
    check_step(cfg, drafter, w, batch, k, requests=[0, B // 2, B - 1], what=f"wide {B}")
    drafter.close()
