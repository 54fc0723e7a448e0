"""The draw of the accept/sample kernel against cumulative sums in 64 bits, at the sizes where its slices, steps and scans end."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def binding():
    from paper_2506_18952_b200 import binding as b
    b.load_library()
    return b


# One CTA of 256 threads, clusters of 2, 4 and 8, one CTA of 1024; a chunk (128 entries) and less, one more than a step of all
# warps, several steps, more than four chunks per lane of the scan (few CTAs per sequence, or a large vocabulary); staged and not;
# rows that start on no 16-byte boundary; more positions than warps.
@pytest.mark.parametrize("B,k,V", [
    (3, 2, 1), (3, 2, 5), (2, 3, 127), (2, 3, 128), (2, 3, 129), (1, 4, 1000), (5, 4, 1921), (40, 2, 3969), (4, 4, 3970), (3, 1, 8064),
    (3, 1, 8192), (9, 3, 8193), (6, 9, 16384), (80, 2, 8000), (80, 40, 2061), (2, 20, 6000), (6, 4, 16388), (2, 20, 20001), (3, 4, 32768), (3, 4, 32896), (30, 2, 33025), (300, 1, 20000),
    (700, 0, 17000), (600, 1, 33000), (2, 2, 140000)])
@pytest.mark.parametrize("q_dtype", [torch.float32, torch.bfloat16])
def test_the_token_is_where_the_cumulative_mass_passes_the_uniform(binding, B, k, V, q_dtype):
    g = torch.Generator(device=DEV).manual_seed(V + B)
    H = 64
    hidden = torch.randn((B, k + 1, H), generator=g, device=DEV).bfloat16()
    W = (torch.randn((V, H), generator=g, device=DEV) * 0.35).bfloat16()
    q = torch.softmax(torch.randn((B, max(k, 1), V), generator=g, device=DEV) * 2.0, 2)[:, :k].to(q_dtype).contiguous()
    tok = torch.randint(0, V, (B, k), generator=g, device=DEV, dtype=torch.int32)
    u = torch.rand((B, k + 1), generator=g, device=DEV)
    u[0, k], u[-1, k] = 0.0, 1.0 - 2.0 ** -24
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_verify(hidden, W, tok, q, u, 0.0, want_logits=True)
        torch.cuda.synchronize()
    assert int(out.status.item()) & ~binding.FLAG_R_ZERO == 0
    at = torch.arange(B, device=DEV)
    n, t = out.accept_len.long(), out.next_tok.long()
    p = torch.softmax(out.logits.double(), 2)
    r = p[at, n]
    if k:
        drafted = torch.where((n < k)[:, None], q.double()[at, n.clamp(max=k - 1)], torch.zeros_like(r))
        r = (r - drafted).clamp(min=0.0)
        r = torch.where(r.sum(1, keepdim=True) > 0, r, p[at, n])
    cum = r.cumsum(1)
    target = u[:, k].double() * cum[:, -1]
    # (p in fp32: relative error of about 1e-6, so that a boundary may lie that far off)
    upto = cum[at, t]
    assert (r[at, t] > 0).all()
    assert (target <= upto + 4e-6).all() and (target >= upto - r[at, t] - 4e-6).all()
