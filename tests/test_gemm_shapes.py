"""The LM-head GEMM at the sizes where its tiling, its passes and its layouts can go wrong: operands whose products and sums
are exact in every weight mode, so that the logits have to be the integers' own, bit for bit, however the work is cut."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda"
MODES = {"bf16": False, "int8": False, "w8a8": True, "w8a16": "a16"}


@pytest.fixture(scope="module")
def binding():
    from paper_2506_18952_b200 import binding as b
    b.load_library()
    return b


def exact_operands(B, k, H, V, seed):
    """Hidden rows and weights that every mode holds exactly (row maxima of 127 steps: quantiser scales are powers of two) and
    whose logits spread over a few units.  The two columns with the maxima meet zeros."""
    g = torch.Generator().manual_seed(seed)
    hid = torch.randint(-6, 7, (B, k + 1, H), generator=g).float()
    W = torch.randint(-5, 6, (V, H), generator=g).float()
    hid[..., 0], hid[..., 1] = 127.0, 0.0
    W[:, 0], W[:, 1] = 0.0, -127.0
    shift = 2.0 ** -round(torch.log2(torch.tensor(float(H))).item() / 2 + 2)
    return hid.bfloat16().to(DEV), (W * shift).bfloat16().to(DEV)


def check_lm_head(binding, mode, B, k, H, V, seed=0, options=()):
    hidden, W = exact_operands(B, k, H, V, seed + H + V)
    want = hidden.double().reshape(-1, H) @ W.double().t()
    w_scale = None
    if mode != "bf16":
        W, w_scale = binding.hola_quantize_w8(W)
    with binding.HolaVerify(B, k, H, V) as ctx:
        for o in options:
            ctx.hola_set_option(*o)
        out = ctx.hola_lm_head_entropy(hidden, W, want_logits=True, w_scale=w_scale, a8=MODES[mode])
        torch.cuda.synchronize()
    assert int(out.status.item()) == 0
    assert torch.equal(out.logits.reshape(-1, V).double(), want)
    # statistics: sums of V positive fp32 terms around the maximum, a few 1e-7 relative each, times |logZ| or H up to 12
    lse = torch.logsumexp(want, 1)
    p = torch.exp(want - lse[:, None])
    H_ref = lse - (p * want).sum(1)
    assert (out.logZ.reshape(-1).double() - lse).abs().max() < 2e-5
    assert (out.entropy.reshape(-1).double() - H_ref).abs().max() < 5e-5


# Rows of 8-bit planes are padded to 128 bytes: H below a block, a tail behind whole blocks, several blocks per ring slot and a
# tail, and no padding at all.
@pytest.mark.parametrize("mode", ["w8a8", "w8a16"])
@pytest.mark.parametrize("B,k,H,V", [(3, 2, 16, 777), (9, 4, 144, 2000), (7, 3, 1040, 5003), (33, 3, 400, 9000), (4, 0, 256, 4097)])
def test_padded_rows_of_eight_bit_planes(binding, mode, B, k, H, V):
    check_lm_head(binding, mode, B, k, H, V)


# Small vocabularies: the rows are cut into several passes over few tiles, all in one launch.  The last pass ends inside a block of
# rows, or holds a single row; tiles of 32, 64, 96 and 128 rows per CTA; a ragged last tile; a partial last K block; with tiles left
# over for some pairs.
@pytest.mark.parametrize("mode,B,k,H,V", [
    ("bf16", 139, 2, 1304, 1272), ("bf16", 128, 3, 512, 2000), ("bf16", 64, 2, 200, 1030), ("bf16", 43, 5, 264, 3001),
    ("bf16", 256, 8, 128, 1003), ("bf16", 129, 0, 4096, 700), ("int8", 29, 8, 944, 2904), ("int8", 97, 0, 2048, 520),
    ("w8a8", 64, 5, 1040, 4000), ("w8a8", 200, 1, 512, 700), ("w8a16", 36, 5, 576, 3550), ("w8a16", 41, 2, 2048, 640)])
def test_rows_of_small_vocabularies_in_several_passes(binding, mode, B, k, H, V):
    wd = {"bf16": binding.HOLA_W_BF16, "int8": binding.HOLA_W_INT8, "w8a8": binding.HOLA_W8A8, "w8a16": binding.HOLA_W8A16}[mode]
    plan = binding.hola_plan_for_shape(148, H, V, B * (k + 1), wd)
    assert plan["passes"] > 1 and plan["kernels_per_call"] == 2
    check_lm_head(binding, mode, B, k, H, V)


# Passes in one launch keep in step by counters, which every launch has to leave at zero for the next: with other numbers of passes
# (None: the plan's own), so of groups, on one context.  They are a pace and nothing else, so the logits alone would not show it.
@pytest.mark.parametrize("mode,B,k,H,V", [
    ("bf16", 300, 3, 64, 30000), ("bf16", 300, 3, 520, 30001), ("int8", 80, 4, 128, 30000), ("w8a8", 200, 4, 128, 40001),
    ("w8a16", 150, 3, 256, 40000), ("mixed", 80, 4, 256, 30000)])
def test_passes_that_keep_step_over_several_tiles_leave_their_counters_clean(binding, mode, B, k, H, V):
    hidden, W = exact_operands(B, k, H, V, 3)
    want = (hidden.double().reshape(-1, H) @ W.double().t()).float()
    scale = None
    if mode == "mixed":
        W = binding.hola_quantize_mixed(W, ([8, 16, 8] * V)[:-(-V // binding.GROUP_ROWS)])
    elif mode != "bf16":
        W, scale = binding.hola_quantize_w8(W)
    code = {"bf16": binding.HOLA_W_BF16, "int8": binding.HOLA_W_INT8, "w8a8": binding.HOLA_W8A8, "w8a16": binding.HOLA_W8A16,
            "mixed": binding.HOLA_W_MIXED}[mode]
    with binding.HolaVerify(B, k, H, V) as ctx:
        assert not ctx.hola_selftest_pace().any()
        for passes in (None, 5, 3, 7):
            if passes:
                ctx.hola_set_option(binding.HOLA_OPT_PASSES, passes)
            plan = ctx.hola_plan(B, k, code)
            groups, tiles = plan["grid"] // (2 * plan["passes"]), -(-V // plan["tile_v"])
            assert plan["passes"] >= 2 and plan["kernels_per_call"] == 2 and tiles > groups
            for _ in range(2):
                out = ctx.hola_lm_head_entropy(hidden, W, want_logits=True, w_scale=scale, a8=MODES.get(mode, False))
                assert torch.equal(out.logits.reshape(-1, V), want)
                assert not ctx.hola_selftest_pace().any()


# Rows that start on no 32-byte sector are copied onto lines where there is enough to do.  `plan`: rows per tile, ring slots, rows per
# pass, passes.  All have a partial last K block: in a slot of its own behind slots of two and of four blocks, or one block per slot
# like the others (rotating units, two MMAs per K step).
@pytest.mark.parametrize("B,k,H,V,plan,copied", [
    (32, 3, 1032, 60000, (208, 4, 128, 1), True),                                                   # two blocks per slot
    (24, 3, 8136, 3000, (64, 4, 96, 1), True), (60, 2, 5320, 1500, (64, 4, 96, 2), True),           # four, in one pass and in two
    (97, 2, 2008, 20003, (256, 4, 336, 1), True), (86, 5, 1544, 19001, (256, 4, 288, 2), True),     # rotating units
    (88, 4, 1032, 20003, (256, 4, 448, 1), True), (125, 7, 520, 40001, (256, 4, 512, 2), True),     # two MMAs
    # rows on sectors (a copy would gain nothing: 37.8 -> 40.4, 31.4 -> 33.1 us); one tile per pair and more than 256 rows
    (39, 7, 592, 53988, (256, 4, 336, 1), False), (74, 4, 1312, 10325, (256, 4, 384, 1), False),
    (60, 7, 2456, 9633, (256, 4, 480, 1), False),
    # too few rows per pass, or too little to do
    (24, 3, 5512, 1000, (128, 4, 32, 3), False), (100, 4, 2056, 700, (128, 8, 64, 8), False),
    (23, 3, 1032, 50003, (240, 4, 96, 1), False), (77, 4, 136, 64001, (256, 4, 416, 1), False)])
def test_rows_copied_onto_lines(binding, B, k, H, V, plan, copied):
    got = binding.hola_plan_for_shape(148, H, V, B * (k + 1))
    assert tuple(got[n] for n in ("tile_v", "stages", "rows_per_pass", "passes")) == plan
    form = binding.hola_hidden_form_for_shape(148, H, V, B * (k + 1))
    assert form == (binding.HOLA_HIDDEN_ON_LINES if copied else binding.HOLA_HIDDEN_IN_PLACE)
    check_lm_head(binding, "bf16", B, k, H, V)


def test_a_copy_of_the_rows_is_a_launch_of_its_own(binding):
    from cuda.bindings import runtime
    for B, k, H, V, mode in [(32, 3, 1032, 60000, "bf16"), (23, 3, 1032, 50003, "bf16"), (9, 4, 144, 2000, "w8a8")]:
        hidden, W = exact_operands(B, k, H, V, 1)
        scale = None
        if mode != "bf16":
            W, scale = binding.hola_quantize_w8(W)
        tok = torch.zeros((B, k), dtype=torch.int32, device=DEV)
        q = torch.full((B, k, V), 1.0 / V, device=DEV)
        u = torch.rand((B, k + 1), device=DEV)
        code = binding.HOLA_W_BF16 if mode == "bf16" else binding.HOLA_W8A8
        with binding.HolaVerify(B, k, H, V) as ctx:
            out = ctx.alloc_outputs(B, k, False)
            graph = torch.cuda.CUDAGraph(keep_graph=True)
            with torch.cuda.graph(graph):
                ctx.hola_verify(hidden, W, tok, q, u, 0.0, out=out, w_scale=scale, a8=MODES[mode])
            err, _, nodes = runtime.cudaGraphGetNodes(runtime.cudaGraph_t(init_value=graph.raw_cuda_graph()), 64)
            assert int(err) == 0
            copied = binding.hola_hidden_form_for_shape(148, H, V, B * (k + 1), code) != binding.HOLA_HIDDEN_IN_PLACE
            assert nodes == ctx.hola_plan(B, k, code)["kernels_per_call"] + copied


@pytest.mark.parametrize("B,k,H,V", [(33, 4, 320, 5001), (50, 2, 136, 9002), (64, 2, 64, 20003)])
def test_statistics_of_an_odd_vocabulary_without_logits(binding, B, k, H, V):
    hidden, W = exact_operands(B, k, H, V, 5)
    want = hidden.double().reshape(-1, H) @ W.double().t()
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_lm_head_entropy(hidden, W)
        torch.cuda.synchronize()
    assert int(out.status.item()) == 0
    assert (out.logZ.reshape(-1).double() - torch.logsumexp(want, 1)).abs().max() < 2e-5
