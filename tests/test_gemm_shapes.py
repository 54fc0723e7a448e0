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
