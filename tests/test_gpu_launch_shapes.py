"""Kernels at the edges of their launch rules: the sizes where one form hands over to another, remainders of tiles, and
several units of work in one thread block.  Each against a plain PyTorch fp32 reference of the same operation."""
import pytest
import torch

import synth_inputs as si
from helpers import PLAN_FLEX, gemm_plan, partial_ranges, rel_err, to_bf16_cuda, weights_to_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    from paper_2512_16483_b200 import binding
    binding.load_library()
    return binding


@pytest.mark.parametrize("B,H,D,r,L", [
    (12, 16, 64, 169, 424),     # more units than SMs; the second tile of every unit is a remainder of 41 rows
    (3, 16, 128, 1600, 300),    # units of two tiles and of one (1600 = 6 * 256 + 64) walked by the same blocks, 3 key blocks
    (5, 16, 128, 700, 129),     # the same with an even number of key blocks, the last with a single key
    (10, 30, 64, 100, 100),     # one key block: set-up, softmax and store of consecutive units only
    (2, 16, 128, 1100, 1500),   # lone tiles walked: 9 tiles a head, the last of 76 rows
    (1, 16, 128, 400, 2921),    # key ranges over a cluster, four tiles, the last of 16 rows
    (1, 3, 128, 5, 6441),       # six ranges, fewer rows than a slice's share for every block
    (16, 16, 64, 100, 600),     # lone tiles walked as two streams of 3 and 2 blocks
    (9, 16, 64, 128, 513),      # the same, a unit a block, the last block with a single key
    (1, 40, 64, 257, 1030),     # pairs whose second unit is one row
    (1, 16, 128, 128, 128), (1, 1, 64, 1, 1),
])
def test_attention_launch_shapes(fv, B, H, D, r, L):
    g = torch.Generator(device="cuda").manual_seed(B * 1000 + r)
    L_cap = (L + 127) // 128 * 128
    q = torch.randn((B, r, H * D), generator=g, device="cuda").bfloat16()
    K = torch.randn((B, H, L_cap, D), generator=g, device="cuda").bfloat16()
    Vt = torch.randn((B, H, D, L_cap), generator=g, device="cuda").bfloat16()
    q[:, ::3] *= 6.0            # rows whose maximum moves: the accumulator is rescaled in some blocks only
    for _ in range(3):          # blocks of work follow one another differently from launch to launch
        out = fv.fvar_attention(q, K, Vt, L)
    assert fv.kernel_poll_status() == fv.OK
    s = torch.einsum("brhd,bhld->bhrl", q.float().view(B, r, H, D), K[:, :, :L].float()) * D ** -0.5
    ref = torch.einsum("bhrl,bhdl->brhd", s.softmax(-1), Vt[..., :L].float()).reshape(B, r, H * D)
    _, cos = rel_err(out.float().cpu().numpy(), ref.cpu().numpy())
    # P and the result are rounded to bf16 (2^-8 of the value at most each); sharp rows are many times the RMS
    bad = (out.float() - ref).abs() - (2.0 ** -6 * ref.abs() + 3e-2 * ref.square().mean().sqrt())
    assert bad.max() <= 0 and cos >= 0.9999, (float(bad.max()), cos)


@pytest.mark.parametrize("V", [8, 1000, 2048, 4104])
def test_transitions_repeat_on_one_context(fv, V):
    """Codeword search in every form its rule takes (1 to 512 rows, few and many codewords); the chain run twice on one
    context gives the same codes, map and tokens, and the codes are those of the fp32 scores."""
    shp, B = si.shape_tiny(n_blocks=1, scales=(1, 2, 3, 8, 16)), 2
    ctx = fv.Fvar(weights_to_cuda(si.make_weights(5, shp)), blocks_per_group=1, n_heads=shp.n_heads, head_dim=shp.head_dim,
                  ffn_dim=shp.ffn_dim, scale_hw=shp.hw(), max_batch=B, ctx_len=0, ctx_width=0)
    Ms, C = shp.tokens_per_scale(), shp.width
    Z = to_bf16_cuda(si.make_codebook(6, V, C))
    ctx.set_codebook(Z)
    got = []
    for _ in range(2):
        run = []
        for k in range(len(Ms)):
            fo = to_bf16_cuda(si.make_step_outputs(7, k, B, Ms[k], si.make_codebook(6, V, C), 0.1))
            codes, nxt = ctx.scale_transition(fo, k, Ms[k + 1] if k + 1 < len(Ms) else None, pairs=True)
            score = fo.float() @ Z.float().T - 0.5 * Z.float().square().sum(-1)
            assert torch.equal(codes.long(), score.argmax(-1)), k
            run += [codes.clone()] + ([nxt.clone()] if nxt is not None else [])
        got.append(run + [ctx.get_feature(B, Ms[-1], C)])
    assert ctx.poll_status() == fv.OK
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("C,hw,B", [
    (640, ((3, 5), (5, 7), (14, 16), (16, 18)), 3),    # long windows, then short ones: both forms; 160 groups of four channels
    (192, ((1, 1), (2, 9), (13, 7), (13, 13)), 2),    # one window for all, a taller and a wider window, equal sizes a side
    (64, ((1, 2), (20, 33), (40, 40)), 1),        # fewer channels than a warp's round
])
def test_down_in_both_forms(fv, C, hw, B):
    """The next tokens are the window means of the accumulated map, whichever form the number of windows picks."""
    shp = si.shape_tiny(n_blocks=1, width=C, n_heads=C // 64, head_dim=64, ffn_dim=64, scale_hw=hw)
    ctx = fv.Fvar(weights_to_cuda(si.make_weights(8, shp)), blocks_per_group=1, n_heads=shp.n_heads, head_dim=64, ffn_dim=64, scale_hw=shp.hw(),
                  max_batch=B, ctx_len=0, ctx_width=0)
    Ms, Z = shp.tokens_per_scale(), si.make_codebook(9, 64, C)
    ctx.set_codebook(to_bf16_cuda(Z))
    for k in range(len(Ms) - 1):
        fo = to_bf16_cuda(si.make_step_outputs(10, k, B, Ms[k], Z, 0.1))
        _, nxt = ctx.scale_transition(fo, k, Ms[k + 1], pairs=True)
        F = ctx.get_feature(B, Ms[-1], C).double().view(B, *hw[-1], C).permute(0, 3, 1, 2)
        pool = torch.nn.functional.adaptive_avg_pool2d
        ref, mag = (pool(x, hw[k + 1]).permute(0, 2, 3, 1).reshape(B, Ms[k + 1], C) for x in (F, F.abs()))
        for half in (0, 1):                       # both branches; bf16 rounding and an fp32 sum over the window
            assert ((nxt[half::2].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * mag).all(), (k, half)
    assert ctx.poll_status() == fv.OK


@pytest.mark.parametrize("R,N,K,width", [
    (33, 64, 64, 32), (400, 192, 2048, 160), (400, 6144, 200, 224),     # half a feature tile, a remainder of one, K not whole blocks
    (255, 1920, 1920, 64), (257, 1920, 128, 256), (1, 256, 4096, 0),    # an odd number of 128-feature halves, one row past a tile
    (5000, 320, 136, 96), (2704, 1024, 1024, 0), (97, 8192, 2048, 0),   # several tiles a pair, the picked widths
    (79, 8192, 2048, 0), (283, 6144, 2048, 0), (3000, 1920, 1920, -176),
    (410, 8192, 2048, -208), (410, 6144, 2048, -144), (283, 8192, 2048, -144),      # negative: picked, and known to be this
    # odd multiples of 16, whose last 32 rows are half the next tile's: full tiles, last tiles of 1, 15, 16, 17, 31 and 47 rows
    (96, 192, 264, 48), (81, 320, 2048, 80), (127, 1920, 200, 112), (160, 64, 1920, 144), (193, 8192, 128, 176),
    (239, 1024, 4096, 208), (5087, 448, 136, 240), (5008, 256, 72, 112), (2704, 2048, 1024, 208),
])
def test_gemm_free_width_pairs(fv, R, N, K, width):
    if width < 0:
        assert gemm_plan(R, N, K) == (PLAN_FLEX, -width)
        width = 0
    g = torch.Generator(device="cuda").manual_seed(R + N + K)
    A = torch.randn((R, K), generator=g, device="cuda").bfloat16()
    W = torch.randn((N, K), generator=g, device="cuda").bfloat16()
    bias = torch.randn((N,), generator=g, device="cuda").bfloat16()
    out = fv.fvar_gemm_bf16_form(A, W, bias, fv.GEMM_FLEX, width)
    assert fv.kernel_poll_status() == fv.OK
    ref = A.double() @ W.double().T + bias.double()
    bound = 1e-5 * (A.double().abs() @ W.double().abs().T).max()
    assert (out.double() - ref).abs().max() <= bound


@pytest.mark.parametrize("shape,B,k,blocks,per_group,bar,ranges", [
    ("d16", 16, 8, 1, 1, 2e-2, 0), ("d16", 2, 7, 1, 1, 2e-2, 0), ("d16", 2, 8, 2, 2, 2e-2, 0), ("narrow", 1, 3, 3, 3, 2e-2, 0),
    ("crossed", 14, 2, 1, 1, 2e-2, 0),                                      # 3584 rows: 208 a tile in every GEMM
    ("infinity", 1, 7, 1, 1, 3e-2, 4), ("infinity", 1, 7, 2, 2, 3e-2, 4),   # a group's last fc2: added up by a pass of its own
    ("infinity", 1, 7, 2, 1, 3e-2, 4),                                      # by the LayerNorm that writes a group's output, 2048 columns
    ("d16", 6, 7, 3, 3, 2e-2, 4), ("wide", 1, 3, 3, 3, 3e-2, 3), ("wide", 1, 3, 2, 1, 3e-2, 3)])
def test_step_epilogues_of_the_free_width_pairs(fv, shape, B, k, blocks, per_group, bar, ranges):
    """Dense blocks at sizes where that form is taken for out-proj and fc2 (2704 rows of 1024 columns), for QKV and fc1 (400 rows
    of 2048) and for every GEMM with a last chunk of 16 rows (3584 of 1024), every epilogue of it and the KV cache against
    the CPU oracle; at 200 and 338 rows of 1024 columns and 324 of 512 fc2 is not split.  With `ranges`, fc2 leaves the sums of
    that many K ranges, which the next block's LayerNorm adds up, within a group and from one dense group to the next, or
    after the last block a kernel of its own: four, or three where K / 64 = 66 is a multiple of 6 and not of 8."""
    import numpy as np
    from oracle import fvar_oracle as orc
    from helpers import assert_close
    shp = {"d16": lambda: si.shape_var_d16(n_blocks=blocks, blocks_per_group=per_group),
           "infinity": lambda: si.shape_infinity_2b(n_blocks=blocks, blocks_per_group=per_group),
           "crossed": lambda: si.shape_tiny(n_blocks=blocks, blocks_per_group=per_group, width=1024, n_heads=16, head_dim=64, ffn_dim=4096, scales=(1, 2, 16, 16), cross=True),
           "narrow": lambda: si.shape_tiny(n_blocks=blocks, blocks_per_group=per_group, width=512, n_heads=8, head_dim=64, ffn_dim=4224, scales=(1, 2, 3, 18, 19)),
           "wide": lambda: si.shape_tiny(n_blocks=blocks, blocks_per_group=per_group, width=2048, n_heads=16, head_dim=128, ffn_dim=4224, scales=(1, 2, 3, 18, 19))}[shape]()
    M, C, F = shp.tokens_per_scale()[k], shp.width, shp.ffn_dim
    assert partial_ranges(B * M, C, F) == ranges
    if shape == "crossed":
        for N, K in ((3 * C, C), (C, C), (F, C), (C, F)):
            assert gemm_plan(B * M, N, K) == (PLAN_FLEX, 208)
    w = si.make_weights(11, shp)
    ctx = fv.Fvar(weights_to_cuda(w), blocks_per_group=per_group, n_heads=shp.n_heads, head_dim=shp.head_dim, ffn_dim=shp.ffn_dim, scale_hw=shp.hw(),
                  max_batch=B, ctx_len=shp.ctx_len, ctx_width=shp.ctx_width)
    o = orc.Oracle(w, shp.n_heads, per_group, shp.hw(), shp.ln_eps)
    cond = si.make_cond(12, B, shp.width)
    text = si.make_context(13, B, shp.ctx_len, shp.ctx_width) if shp.has_cross_attn else None
    ctx.set_cond(to_bf16_cuda(cond), to_bf16_cuda(text) if text is not None else None)
    o.set_cond(cond, text)
    for scale in (k, k):                # the second time over the keys and values the first one left in the cache
        toks = si.make_tokens(14, B, M, shp.width)
        ctx.scale_step(to_bf16_cuda(toks), scale)
        o.scale_step(toks, scale, orc.Policy("dense", "pair"))
        for g in range(shp.n_groups):
            assert_close(ctx.get_group_output(g, M).cpu().numpy(), np.stack([o.group_cache[g][b] for b in range(B)]), max_rel=bar, what="%s, group %d" % (shape, g))
        ctx.kv_append(scale)
        o.kv_append(scale)
    assert ctx.poll_status() == fv.OK


@pytest.mark.parametrize("form,R,N,K", [("GEMM_SKINNY", 16, 8192, 2048), ("GEMM_KSPLIT", 100, 2048, 8192), ("GEMM_FLEX", 400, 8192, 2048),
                                        ("GEMM_SINGLE", 100, 8192, 2048), ("GEMM_PAIR", 400, 8192, 2048)])
def test_gemm_waits_for_a_weight_that_the_call_before_writes(fv, form, R, N, K):
    """The second operand comes from the library call just before, which lets its successor start early: every form
    has to read it after that call has ended."""
    g = torch.Generator(device="cuda").manual_seed(R + N)
    A = torch.randn((R, K), generator=g, device="cuda").bfloat16()
    pair = torch.randn((2, N, K), generator=g, device="cuda").bfloat16()
    for s in (1.0, 0.0, -1.0, 2.0, 1.0, 0.0):          # the buffer of the weight is reused: it holds an earlier one
        W = fv.fvar_cfg_combine(pair, s)
        out = fv.fvar_gemm_bf16_form(A, W[0], None, getattr(fv, form), 0)
        ref = A.double() @ W[0].double().T
        bound = 1e-5 * (A.double().abs() @ W[0].double().abs().T).max()       # fp32 sums of at most 8192 products
        del W
        assert (out.double() - ref).abs().max() <= bound, s
    assert fv.kernel_poll_status() == fv.OK


def _join_calls(fv):
    """Every way the library launches a kernel, as calls on the current stream."""
    g = torch.Generator(device="cuda").manual_seed(3)
    def rnd(*shape): return torch.randn(shape, generator=g, device="cuda")
    A, W = {R: rnd(R, 512).bfloat16() for R in (16, 200)}, rnd(256, 512).bfloat16()
    x, vec, prev, pair = rnd(2, 64, 256), rnd(2, 256), rnd(2, 16, 256), rnd(2, 64, 256).bfloat16()
    scores, out = rnd(2, 64), rnd(2, 64, 256)
    def attn(r, L):
        q, K, Vt = rnd(1, r, 128).bfloat16(), rnd(1, 1, L, 128).bfloat16(), rnd(1, 1, 128, L).bfloat16()
        return lambda: fv.fvar_attention(q, K, Vt, L)
    calls = {"form %s" % f: (lambda f=f, R=R: fv.fvar_gemm_bf16_form(A[R], W, None, getattr(fv, f), 0))
             for f, R in (("GEMM_SINGLE", 200), ("GEMM_PAIR", 200), ("GEMM_SKINNY", 16), ("GEMM_KSPLIT", 200), ("GEMM_FLEX", 200))}
    return dict(calls, attention=attn(64, 128), ranges=attn(16, 4096), scores=lambda: fv.fvar_row_scores(x), select=lambda: fv.fvar_select_topr(scores, 9)[0],
                ln=lambda: fv.fvar_ln_modulate(x, vec, vec, 1e-6), fill=lambda: fv.fvar_rtr_fill(prev, (4, 4), (8, 8), None, out),
                combine=lambda: fv.fvar_cfg_combine(pair, 2.0))


def _edge_types(graph):
    """{(from, to): type} of a captured graph; type 1 is a programmatic edge, 0 a full one."""
    import ctypes as ct

    class Edge(ct.Structure):
        _fields_ = [("from_port", ct.c_ubyte), ("to_port", ct.c_ubyte), ("type", ct.c_ubyte), ("reserved", ct.c_ubyte * 5)]
    ask, g, n = ct.CDLL("libcuda.so.1").cuGraphGetEdges_v2, ct.c_void_p(graph.raw_cuda_graph()), ct.c_size_t(0)
    assert ask(g, None, None, None, ct.byref(n)) == 0
    fr, to, data = (ct.c_void_p * n.value)(), (ct.c_void_p * n.value)(), (Edge * n.value)()
    assert ask(g, fr, to, data, ct.byref(n)) == 0
    return {(a, b): e.type for a, b, e in zip(fr, to, data)}


def test_a_launch_where_branches_of_a_capture_meet_waits_for_all_of_them(fv):
    """A kernel that depends on several others starts when they have ended; one that follows a single kernel may start
    early.  The step's own graphs are captured through the same launches."""
    x, pair = torch.randn(2, 64, 256, device="cuda"), torch.randn(2, 64, 256, device="cuda").bfloat16()
    for name, call in _join_calls(fv).items():
        ref = call().clone()
        fv.fvar_row_scores(x), fv.fvar_cfg_combine(pair, 1.0)
        main, side, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=main):
            keep = [fv.fvar_row_scores(x)]
            side.wait_stream(main)
            with torch.cuda.stream(side):
                keep += [fv.fvar_cfg_combine(pair, 1.0)]
            keep += [fv.fvar_cfg_combine(pair, 1.0)]
            main.wait_stream(side)
            got = call()
        edges = _edge_types(graph)
        last = [b for _, b in edges]
        meet = [t for (_, b), t in edges.items() if last.count(b) > 1]
        assert meet == [0, 0], (name, edges)
        assert [t for (_, b), t in edges.items() if last.count(b) == 1] == [1, 1], (name, edges)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, ref), name
    assert fv.kernel_poll_status() == fv.OK
