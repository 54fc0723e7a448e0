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
# over for some pairs (the calls come twice: what the groups of pairs keep step by has to be as it was).
@pytest.mark.parametrize("mode,B,k,H,V", [
    ("bf16", 139, 2, 1304, 1272), ("bf16", 128, 3, 512, 2000), ("bf16", 64, 2, 200, 1030), ("bf16", 43, 5, 264, 3001),
    ("bf16", 256, 8, 128, 1003), ("bf16", 129, 0, 4096, 700), ("int8", 29, 8, 944, 2904), ("int8", 97, 0, 2048, 520),
    ("w8a8", 64, 5, 1040, 4000), ("w8a8", 200, 1, 512, 700), ("w8a16", 36, 5, 576, 3550), ("w8a16", 41, 2, 2048, 640)])
def test_rows_of_small_vocabularies_in_several_passes(binding, mode, B, k, H, V):
    wd = {"bf16": binding.HOLA_W_BF16, "int8": binding.HOLA_W_INT8, "w8a8": binding.HOLA_W8A8, "w8a16": binding.HOLA_W8A16}[mode]
    plan = binding.hola_plan_for_shape(148, H, V, B * (k + 1), wd)
    assert plan["passes"] > 1 and plan["kernels_per_call"] == 2
    check_lm_head(binding, mode, B, k, H, V)


@pytest.mark.parametrize("mode,B,k,H,V", [("bf16", 300, 3, 64, 30000), ("w8a8", 200, 4, 128, 40001)])
def test_passes_that_keep_step_over_several_tiles_leave_their_counters_clean(binding, mode, B, k, H, V):
    hidden, W = exact_operands(B, k, H, V, 3)
    want = (hidden.double().reshape(-1, H) @ W.double().t()).float()
    scale = None
    if mode != "bf16":
        W, scale = binding.hola_quantize_w8(W)
    with binding.HolaVerify(B, k, H, V) as ctx:
        for _ in range(3):
            out = ctx.hola_lm_head_entropy(hidden, W, want_logits=True, w_scale=scale, a8=MODES[mode])
            assert torch.equal(out.logits.reshape(-1, V), want)


# Rows that start on no 128-byte line are copied onto lines where there is enough to do: a partial last K block and several per ring
# slot, four tiles per pair, several passes, rotating units, two MMAs per K step; the last one stays as it is.  An odd vocabulary:
# 16-byte stores of logits end within the row's pitch.
@pytest.mark.parametrize("B,k,H,V", [(24, 3, 5512, 1000), (32, 3, 1032, 60000), (100, 4, 2056, 700), (97, 2, 2008, 20003), (86, 5, 1544, 19001), (24, 3, 5128, 1000)])
def test_rows_copied_onto_lines(binding, B, k, H, V):
    check_lm_head(binding, "bf16", B, k, H, V)


@pytest.mark.parametrize("B,k,H,V", [(33, 4, 320, 5001), (50, 2, 136, 9002), (64, 2, 64, 20003)])
def test_statistics_of_an_odd_vocabulary_without_logits(binding, B, k, H, V):
    hidden, W = exact_operands(B, k, H, V, 5)
    want = hidden.double().reshape(-1, H) @ W.double().t()
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_lm_head_entropy(hidden, W)
        torch.cuda.synchronize()
    assert int(out.status.item()) == 0
    assert (out.logZ.reshape(-1).double() - torch.logsumexp(want, 1)).abs().max() < 2e-5
