"""GPU parity of the mixed-width LM head (groups of 256 vocabulary rows at 4, 8 or 16 bits, HOLA_W_MIXED) and of the
4-bit quantiser kernel, against oracle/lobi.py and the fp64 verify oracle on the dequantised matrix."""
import numpy as np
import pytest
import torch

from oracle import compare, lobi, ref
from paper_2506_18952_b200 import workloads

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def binding():
    from paper_2506_18952_b200 import binding as b
    b.load_library()
    return b


def _np(t):
    return compare.torch_to_numpy(t)


def _widths(V, pattern):
    ng = -(-V // 256)
    return [pattern[g % len(pattern)] for g in range(ng)]


@pytest.mark.parametrize("V,H", [(300, 128), (1000, 512), (4099, 256)])
def test_w4_quantiser_is_bit_exact(binding, V, H):
    g = torch.Generator(device=DEV).manual_seed(V + H)
    W = (torch.randn((V, H), generator=g, device=DEV) * 0.02).bfloat16()
    W[:, 128:256] *= 0.05 if H >= 256 else 1.0          # a quiet sub-block: smaller exponents
    W[3] = 0                                            # an all-zero row
    W[5] = 0
    W[5, 0] = 0.4375                                    # 112 * 2^-8: scale 2^-8, ties at half steps below
    W[5, 1:4] = torch.tensor([0.03125 * 0.5, 0.03125 * 1.5, -0.03125 * 2.5], device=DEV).bfloat16()
    lib = binding.load_library()
    packed = torch.empty((V, H // 2), dtype=torch.uint8, device=DEV)
    shifts = torch.full((H // 128, V), 255, dtype=torch.uint8, device=DEV)
    scale = torch.empty((V,), dtype=torch.float32, device=DEV)
    import ctypes
    st = lib.hola_quantize_w4(ctypes.c_void_p(W.data_ptr()), V, H, ctypes.c_void_p(packed.data_ptr()),
                              ctypes.c_void_p(shifts.data_ptr()), V, ctypes.c_void_p(scale.data_ptr()), None)
    assert st == 0
    torch.cuda.synchronize()
    c, e, s = lobi.quantize_rows_w4(W.float().cpu().numpy())
    assert np.array_equal(_np(scale), s)
    assert np.array_equal(_np(shifts).T, e)
    assert np.array_equal(_np(packed), lobi.pack_nibbles(c))
    assert lib.hola_quantize_w4(ctypes.c_void_p(W.data_ptr()), V, 100, ctypes.c_void_p(packed.data_ptr()),
                                ctypes.c_void_p(shifts.data_ptr()), V, ctypes.c_void_p(scale.data_ptr()), None) == 2


def _mixed_oracle(w, widths, **kw):
    hid = ref.bf16_bits_to_f64(_np(w.hidden))
    Wd = lobi.dequantize_mixed(ref.bf16_bits_to_f64(_np(w.W_lm)).astype(np.float32), widths)
    return ref.verify(hid, Wd, _np(w.draft_tok), _np(w.draft_q), _np(w.uniforms), w.tau, keep_logits=True, **kw)


@pytest.mark.parametrize("B,k,H,V,pattern", [
    (1, 4, 128, 1000, [16, 4, 8, 4]),          # the tiny batch: four groups, every width, ragged last group
    (9, 3, 256, 700, [4, 8, 16]),              # three groups, two sub-blocks per row
    (37, 6, 256, 5000, [8, 8, 4, 16, 8]),      # 259 rows: two passes over the head
    (20, 3, 384, 2048, [4]),                   # every group at 4 bits, whole groups only
    (6, 2, 128, 3001, [16, 8]),                # no 4-bit group at all
])
def test_mixed_width_head_matches_oracle_on_the_dequantised_matrix(binding, B, k, H, V, pattern):
    w = workloads.gaussian_head("mixed", B, k, H, V, seed=B + V, device=DEV, w_std=0.3, sigma=1.0, tau=1.5 + 0.1 * k,
                                sigma_far=0.2)
    widths = _widths(V, pattern)
    head = binding.hola_quantize_mixed(w.W_lm, widths)
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True)
        torch.cuda.synchronize()
    assert int(out.status.item()) & binding.FLAG_TIMEOUT == 0
    orc = _mixed_oracle(w, widths)
    rep = compare.compare(orc, _np(w.draft_q), _np(w.uniforms), _np(out.accept_len), _np(out.next_tok),
                          _np(out.entropy), _np(out.logZ), _np(out.logits))
    print(rep.summary())
    assert rep.ok, rep.summary()
    assert rep.accept_margin_cases <= max(1, B // 20) and rep.token_margin_cases <= max(1, B // 10)


def test_mixed_width_integer_weights_are_bit_exact(binding):
    """Weights that are of the stored forms already (4-bit: c << e with a 112 per row; 8-bit: integers with a 127 per
    row; 16-bit: small integers) and small-integer hidden rows: every product and sum is exact, so the logits must
    equal the integer matrix product."""
    g = torch.Generator().manual_seed(4)
    V, H, B, k = 768, 256, 4, 2
    W = torch.zeros((V, H))
    c = torch.randint(-7, 8, (256, 2, 128), generator=g)
    e = torch.randint(0, 5, (256, 2), generator=g)
    c[:, :, 0] = 7
    e[:, 0] = 4
    W[0:256] = (c * (2 ** e)[:, :, None]).reshape(256, H).float()          # group 0: 4 bits
    W[256:512] = torch.randint(-127, 128, (256, H), generator=g).float()   # group 1: 8 bits
    W[256:512, 0] = 127
    W[512:768] = torch.randint(-8, 9, (256, H), generator=g).float()       # group 2: 16 bits
    hidden = torch.randint(-2, 3, (B, k + 1, H), generator=g).float()
    want = (hidden.reshape(-1, H).double() @ W.double().T).reshape(B, k + 1, V)
    q = torch.full((B, k, V), 1.0 / V)
    tok = torch.randint(0, V, (B, k), generator=g, dtype=torch.int32)
    u = torch.rand((B, k + 1), generator=g)
    head = binding.hola_quantize_mixed(W.bfloat16().to(DEV), [4, 8, 16])
    assert torch.all(head.w_scale == 1.0)
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_verify(hidden.bfloat16().to(DEV), head, tok.to(DEV), q.to(DEV), u.to(DEV), 0.0, want_logits=True)
        torch.cuda.synchronize()
    assert torch.equal(out.logits.cpu().double(), want)


def test_mixed_width_arguments_are_validated(binding):
    w = workloads.gaussian_head("mixed-args", 2, 2, 128, 600, seed=3, device=DEV, w_std=0.3)
    with pytest.raises(binding.HolaError):
        binding.hola_quantize_mixed(w.W_lm, [4, 8])                 # three groups, two widths
    with pytest.raises(binding.HolaError):
        binding.hola_quantize_mixed(w.W_lm, [4, 8, 5])
    head = binding.hola_quantize_mixed(w.W_lm, [4, 8, 16])
    assert head.weight_bytes() < w.W_lm.numel() * 2
    with binding.HolaVerify(2, 2, 128, 600) as ctx:
        with pytest.raises(binding.HolaError):
            ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, a8=True)
    with binding.HolaVerify(2, 2, 128, 856) as ctx:                 # a head of another vocabulary size
        with pytest.raises(binding.HolaError):
            ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau)


@pytest.mark.parametrize("name", ["edge", "large_vocab_b32"])
def test_mixed_width_on_the_bandwidth_bound_shapes(binding, name):
    """Full size, widths in the proportions the paper reports (most groups at 8 bits, some at 4, a few kept at 16);
    sampled sequences against the oracle on the dequantised matrix."""
    w = workloads.make_config(name, DEV)
    ng = -(-w.V // 256)
    rng = np.random.default_rng(11)
    widths = rng.choice([4, 8, 16], size=ng, p=[0.2, 0.7, 0.1]).tolist()
    head = binding.hola_quantize_mixed(w.W_lm, widths)
    with binding.HolaVerify(w.B, w.k, w.H, w.V) as ctx:
        out = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True)
        torch.cuda.synchronize()
    assert int(out.status.item()) & binding.FLAG_TIMEOUT == 0
    seqs = list(range(w.B)) if w.B <= 4 else [0, 9, 20, 31]
    sub = w.slice(seqs)
    orc = _mixed_oracle(sub, widths)
    pick = torch.as_tensor(seqs, device=DEV)
    rep = compare.compare(orc, _np(sub.draft_q), _np(sub.uniforms), _np(out.accept_len[pick]), _np(out.next_tok[pick]),
                          _np(out.entropy[pick]), _np(out.logZ[pick]), _np(out.logits[pick]))
    print(name, rep.summary())
    assert rep.ok, rep.summary()


def test_converter_group_size_changes_speed_not_results(binding):
    """The number of converter warps that share a K block is a speed knob: the expansion is exact whoever does it, so
    every setting gives the same logits bit for bit (few K blocks, many K blocks, more groups than ring slots in use)."""
    for B, k, H, V in ((3, 2, 128, 1300), (40, 4, 1024, 2600)):
        w = workloads.gaussian_head("conv-group", B, k, H, V, seed=V, device=DEV, w_std=0.3, sigma=1.0, tau=1.7)
        head = binding.hola_quantize_mixed(w.W_lm, _widths(V, [4, 8, 16, 8, 4]))
        with binding.HolaVerify(B, k, H, V) as ctx:
            base = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True)
            torch.cuda.synchronize()
            assert int(base.status.item()) == 0
            for G in (1, 2, 3, 4, 8, 0):
                ctx.hola_set_option(binding.HOLA_OPT_CONVERTER_GROUP, G)
                out = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True)
                torch.cuda.synchronize()
                assert int(out.status.item()) == 0, G
                assert torch.equal(out.logits, base.logits), G
                assert torch.equal(out.accept_len, base.accept_len) and torch.equal(out.next_tok, base.next_tok)
            for bad in (-1, 9):
                with pytest.raises(binding.HolaError):
                    ctx.hola_set_option(binding.HOLA_OPT_CONVERTER_GROUP, bad)
            # fewer ring slots than groups of converter warps: only as many groups as slots take part
            for slots, G in ((2, 1), (3, 2), (2, 4)):
                ctx.hola_set_option(binding.HOLA_OPT_RING_SLOTS, slots)
                ctx.hola_set_option(binding.HOLA_OPT_CONVERTER_GROUP, G)
                assert ctx.hola_plan(B, k, binding.HOLA_W_MIXED)["stages"] == slots
                out = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True)
                torch.cuda.synchronize()
                assert int(out.status.item()) == 0, (slots, G)
                assert torch.equal(out.logits, base.logits), (slots, G)
    orc = _mixed_oracle(w, _widths(V, [4, 8, 16, 8, 4]))
    rep = compare.compare(orc, _np(w.draft_q), _np(w.uniforms), _np(base.accept_len), _np(base.next_tok),
                          _np(base.entropy), _np(base.logZ), _np(base.logits))
    assert rep.ok, rep.summary()


@pytest.mark.parametrize("B,k,H,V,pattern", [
    (32, 3, 128, 1100, [4, 8]),                # 128 rows, one K block of codes per tile, four operand slots
    (43, 2, 384, 2100, [16, 4, 8]),            # 129 rows: wider accumulators, two operand slots
    (64, 2, 640, 2500, [8, 16, 4, 4]),         # 192 rows, the most one pass holds; an odd number of K blocks
    (193, 0, 256, 900, [4, 16]),               # 193 rows: two passes
    (8, 3, 1408, 5000, [8, 4, 16]),            # 32 rows, the most that four epilogue warps serve: three converter groups
    (11, 2, 384, 40000, [4, 8, 8, 16]),        # 33 rows: two groups again; three tiles per pair
    (1, 4, 2176, 60000, [8, 16, 4]),           # one sequence, several tiles of every width per pair
    (3, 4, 176, 1100, None), (64, 2, 112, 37000, None),   # all 8-bit (no width table): ragged last K block, many tiles
])
def test_expansion_at_the_edges_of_its_tiles(binding, B, k, H, V, pattern):
    """Row counts around the switch of the accumulator layout and of the pass count, K extents around the 128-channel
    blocks of codes and the 64-channel blocks of 16-bit rows: logits against an fp64 product of the dequantised weights
    (fp32 accumulation, one rounding or truncation of 2^-23 per step of sixteen products and per product within a step:
    an error below (H / 16 + 16) 2^-23 of sum |terms|)."""
    w = workloads.gaussian_head("edges", B, k, H, V, seed=B + H, device=DEV, w_std=0.3)
    if pattern is None:
        head, scale = binding.hola_quantize_w8(w.W_lm)
        Wd = head.double() * scale.double()[:, None]
    else:
        head, scale = binding.hola_quantize_mixed(w.W_lm, _widths(V, pattern)), None
        W32 = ref.bf16_bits_to_f64(_np(w.W_lm)).astype(np.float32)
        Wd = torch.from_numpy(lobi.dequantize_mixed(W32, _widths(V, pattern))).to(DEV)
    with binding.HolaVerify(B, k, H, V) as ctx:
        out = ctx.hola_verify(w.hidden, head, w.draft_tok, w.draft_q, w.uniforms, w.tau, want_logits=True, w_scale=scale)
        torch.cuda.synchronize()
    assert int(out.status.item()) == 0
    h = w.hidden.double()
    want = h @ Wd.T
    bound = (H / 16 + 16) * 2.0 ** -23 * (h.abs() @ Wd.abs().T)
    assert torch.all((out.logits.double() - want).abs() <= bound)


@pytest.mark.parametrize("V,H", [(257, 128), (600, 4096), (1025, 4224), (523, 640)])
def test_whole_head_quantiser_is_bit_exact(binding, V, H):
    """One launch for all groups: codes, exponents, scales and copied rows against the oracle, at the edges of what a warp
    keeps in registers (4096 channels), with ragged last groups and rows of zeros, ties and a lone large entry."""
    g = torch.Generator(device=DEV).manual_seed(V)
    W = (torch.randn((V, H), generator=g, device=DEV) * 0.02).bfloat16()
    W[7] = 0
    W[9] = (torch.randint(-254, 255, (H,), generator=g, device=DEV) * 0.5).bfloat16()      # halves of the 8-bit step
    W[9, 0] = 127
    W[11, 5] = 30.0
    W[13] *= 2.0 ** -100                                # steps at the end of the fp32 range
    W[min(270, V - 1)] *= 2.0 ** -100
    widths = _widths(V, [8, 4, 16, 4])
    head = binding.hola_quantize_mixed(W, widths)
    torch.cuda.synchronize()
    W32 = W.float().cpu().numpy()
    at = {4: 0, 8: 0, 16: 0}
    for gi, wd in enumerate(widths):
        lo, hi = 256 * gi, min(V, 256 * gi + 256)
        r = slice(at[wd], at[wd] + hi - lo)
        at[wd] += hi - lo
        scale = _np(head.w_scale[lo:hi])
        if wd == 16:
            assert torch.equal(head.W16[r], W[lo:hi]) and np.all(scale == 1.0)
        elif wd == 8:
            q, s = lobi.quantize_rows_int8(W32[lo:hi])
            assert np.array_equal(_np(head.W8[r]), q) and np.array_equal(scale, s)
        else:
            c, e, s = lobi.quantize_rows_w4(W32[lo:hi])
            assert np.array_equal(_np(head.W4[r]), lobi.pack_nibbles(c)) and np.array_equal(scale, s)
            assert np.array_equal(_np(head.shift4[:, r]).T, e)


@pytest.mark.parametrize("V,H,offset", [(33, 203, 0), (40, 256, 1)])
def test_quantisers_take_rows_that_16_byte_pieces_do_not_tile(binding, V, H, offset):
    g = torch.Generator(device=DEV).manual_seed(H)
    flat = (torch.randn(V * H + 8, generator=g, device=DEV) * 0.02).bfloat16()
    W = flat[offset:offset + V * H].view(V, H)
    W32 = W.float().cpu().numpy()
    q, s = binding.hola_quantize_w8(W)
    q0, s0 = lobi.quantize_rows_int8(W32)
    assert np.array_equal(_np(q), q0) and np.array_equal(_np(s), s0)
    if H % 128 == 0:
        head = binding.hola_quantize_mixed(W, [4])
        c, e, s = lobi.quantize_rows_w4(W32)
        assert np.array_equal(_np(head.W4), lobi.pack_nibbles(c)) and np.array_equal(_np(head.w_scale), s)
        assert np.array_equal(_np(head.shift4).T, e)
        assert torch.equal(binding.hola_quantize_mixed(W, [16]).W16, W)


def test_quantisers_round_every_quotient_of_two_bf16_mantissas_like_the_division(binding):
    """The integers depend on the mantissas of a row's maximum and of an entry, their exponents' difference and the sign:
    128 rows, one per mantissa of the maximum, with every other bf16 value down to 2^-15 of it, in an order in which the
    4-bit sub-blocks take every exponent and in a shuffled one."""
    m = torch.arange(128, 256, dtype=torch.float32)
    mags = torch.cat([m * 2.0 ** -(9 + e) for e in range(16)])                # descending binades below 2^-1
    signs = 1.0 - 2.0 * (torch.arange(mags.numel()) % 2)
    row = torch.cat([mags * signs, -mags * signs])                            # 4096 entries, both signs
    shuffled = row[torch.randperm(row.numel(), generator=torch.Generator().manual_seed(3))]
    W = torch.zeros((256, row.numel()))
    for i in range(128):
        top = m[i] * 2.0 ** -9
        for k, r in enumerate((row, shuffled)):
            W[2 * i + k] = torch.where(r.abs() <= top, r, r * 2.0 ** -8)
            W[2 * i + k, 17] = top
    W = W.bfloat16().to(DEV)
    W32 = W.float().cpu().numpy()
    q, s = binding.hola_quantize_w8(W)
    q0, s0 = lobi.quantize_rows_int8(W32)
    assert np.array_equal(_np(q), q0) and np.array_equal(_np(s), s0)
    head = binding.hola_quantize_mixed(W, [4])
    c, e, s = lobi.quantize_rows_w4(W32)
    assert np.array_equal(_np(head.W4), lobi.pack_nibbles(c)) and np.array_equal(_np(head.shift4).T, e)
    assert set(np.unique(e)) == {0, 1, 2, 3, 4}
    # hidden rows in one and in two planes: an identity-like head of ones picks single entries out as logits
    q8 = torch.zeros((W.shape[1], W.shape[1]), dtype=torch.int8, device=DEV)
    q8.fill_diagonal_(1)
    ones = torch.ones(W.shape[1], dtype=torch.float32, device=DEV)
    hidden = W.view(256, 1, -1)
    with binding.HolaVerify(256, 0, W.shape[1], W.shape[1]) as ctx:
        one = ctx.hola_lm_head_entropy(hidden, q8, w_scale=ones, a8=True).logits[:, 0]
        two = ctx.hola_lm_head_entropy(hidden, q8, w_scale=ones, a8="a16").logits[:, 0]
        torch.cuda.synchronize()
    s1 = torch.from_numpy(s0).to(DEV)[:, None]
    assert torch.equal(one, torch.from_numpy(q0).to(DEV).float() * s1)
    p1, p2, sa, sb = (torch.from_numpy(np.asarray(x)).to(DEV) for x in lobi.quantize_rows_two_plane(W32))
    want = p1.double() * sa.double()[:, None] + p2.double() * sb.double()[:, None]
    assert torch.all((two.double() - want).abs() <= 2.0 ** -22 * want.abs() + 1e-30)       # one fused multiply-add
    assert torch.equal(((two - p1.float() * sa[:, None]) / sb[:, None]).round(), p2.float())


def test_a_head_quantised_anew_into_the_same_buffers_is_the_one_that_is_used(binding):
    """Other widths into the same (large enough) buffers, on one context: the same logits as a head in buffers of its own."""
    import ctypes
    B, k, H, V = 3, 2, 256, 1000
    w = workloads.gaussian_head("anew", B, k, H, V, seed=8, device=DEV, w_std=0.3)
    lib = binding.load_library()
    buf = dict(W16=torch.empty((V, H), dtype=torch.bfloat16, device=DEV), W8=torch.empty((V, H), dtype=torch.int8, device=DEV),
               W4=torch.empty((V, H // 2), dtype=torch.uint8, device=DEV),
               shift4=torch.empty((H // 128 * V,), dtype=torch.uint8, device=DEV))
    scale = torch.empty((V,), dtype=torch.float32, device=DEV)
    with binding.HolaVerify(B, k, H, V) as ctx:
        for widths in ([8, 16, 4, 8], [4, 8, 8, 16], [8, 8, 8, 4], [16, 4, 8, 4]):
            own = binding.hola_quantize_mixed(w.W_lm, widths)
            st = binding.hola_wmix()
            for name, t in buf.items():
                setattr(st, name, t.data_ptr())
            st.group_width, st.group_row = own.group_width.data_ptr(), own.group_row.data_ptr()
            st.rows16, st.rows8, st.rows4 = own.struct.rows16, own.struct.rows8, own.struct.rows4
            assert lib.hola_quantize_mixed(ctypes.c_void_p(w.W_lm.data_ptr()), V, H, ctypes.byref(st),
                                           ctypes.c_void_p(scale.data_ptr()), None) == 0
            head = binding.MixedHead(V, H, widths, buf["W16"], buf["W8"], buf["W4"], buf["shift4"], scale, own.group_width,
                                     own.group_row, st)
            got = ctx.hola_lm_head_entropy(w.hidden, head)
            with binding.HolaVerify(B, k, H, V) as other:
                want = other.hola_lm_head_entropy(w.hidden, own)
                torch.cuda.synchronize()
            assert int(got.status.item()) == 0
            assert torch.equal(got.logits, want.logits), widths


def test_quantiser_takes_an_empty_head_and_any_object_with_a_cuda_stream(binding):
    import types
    empty = binding.hola_quantize_mixed(torch.empty((0, 128), dtype=torch.bfloat16, device=DEV), [])
    assert empty.V == 0 and empty.weight_bytes() == 0 and empty.group_width.numel() == 0 and empty.group_row.numel() == 0
    g = torch.Generator(device=DEV).manual_seed(1)
    W = torch.randn((700, 256), generator=g, device=DEV).bfloat16()
    want = binding.hola_quantize_mixed(W, [4, 8, 16])
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for stream in (side, types.SimpleNamespace(cuda_stream=side.cuda_stream)):
        got = binding.hola_quantize_mixed(W, [4, 8, 16], stream=stream)
        side.synchronize()
        for name in ("W16", "W8", "W4", "shift4", "w_scale", "group_width", "group_row"):
            assert torch.equal(getattr(got, name), getattr(want, name)), name


@pytest.mark.parametrize("groups,rest,H,pattern", [
    (1, 256, 128, [4]), (2, 44, 128, [16, 4]), (16, 256, 128, [8, 4, 16]), (17, 1, 256, [4, 8, 8, 16, 4]),
    (33, 255, 384, [16]), (100, 100, 1152, [8, 16, 8, 4, 4]), (2048, 256, 128, [8, 4, 16, 8]),
    (2049, 3, 128, [4, 16, 8]),                          # more groups than launch parameters hold: through the tables
])
def test_widths_as_launch_parameters_give_the_head_that_tables_give(binding, monkeypatch, groups, rest, H, pattern):
    V = 256 * (groups - 1) + rest
    g = torch.Generator(device=DEV).manual_seed(groups)
    W = (torch.randn((V, H), generator=g, device=DEV) * 0.02).bfloat16()
    widths = _widths(V, pattern)
    assert binding._host is not None
    got = [binding.hola_quantize_mixed(W, x) for x in (widths, tuple(widths))]
    monkeypatch.setattr(binding, "_host", None)
    want = binding.hola_quantize_mixed(W, widths)
    torch.cuda.synchronize()
    for head in got:
        assert (head.V, head.H, head.widths) == (V, H, widths)
        for name in ("W16", "W8", "W4", "shift4", "w_scale", "group_width", "group_row"):
            a, b = getattr(head, name), getattr(want, name)
            assert (a is None and b is None) or (a.dtype == b.dtype and torch.equal(a, b)), name
        for name in ("rows16", "rows8", "rows4"):
            assert getattr(head.struct, name) == getattr(want.struct, name)


def test_widths_on_the_host_are_checked(binding):
    import ctypes
    lib = binding.load_library()
    W = torch.zeros((600, 128), dtype=torch.bfloat16, device=DEV)
    head = binding.hola_quantize_mixed(W, [4, 8, 16])

    def status(widths, V=600, H=128):
        return lib.hola_quantize_mixed_widths(ctypes.c_void_p(W.data_ptr()), V, H, bytes(widths), ctypes.byref(head.struct),
                                              ctypes.c_void_p(head.w_scale.data_ptr()), None)
    assert status([4, 8, 16]) == 0
    assert status([4, 8, 5]) == 1 and status([4, 16, 8]) == 1 and status([8, 4, 16], V=599) == 1     # row counts that do not fit
    assert status([4, 8, 16], H=100) == 2 and lib.hola_quantize_mixed_widths(None, 600, 128, None, None, None, None) == 1
    assert status([4] * 2049, V=2049 * 256) == 2
    torch.cuda.synchronize()


def test_a_list_of_widths_that_changes_during_the_call_leaves_the_head_as_it_was_made(binding, monkeypatch):
    """The native quantiser call lets other threads run; one of them may reuse the list."""
    import ctypes
    lib = binding.load_library()
    W = torch.zeros((600, 128), dtype=torch.bfloat16, device=DEV)
    widths = [4, 8, 16]

    def entry(*args):
        widths[:] = [16, 16]
        return lib.hola_quantize_mixed_widths(*args)
    p = ctypes.c_void_p
    fn = ctypes.CFUNCTYPE(ctypes.c_int, p, ctypes.c_int, ctypes.c_int, p, ctypes.POINTER(binding.hola_wmix), p, p)(entry)
    monkeypatch.setitem(binding._entry, "hola_quantize_mixed_widths", ctypes.cast(fn, p).value)
    head = binding.hola_quantize_mixed(W, widths)
    torch.cuda.synchronize()
    assert widths == [16, 16] and head.widths == [4, 8, 16] and head.group_width.tolist() == [4, 8, 16]
