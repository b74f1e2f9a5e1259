"""Every kernel variant at the sizes where its split of the work can go wrong: one row and one channel more than a tile,
remainders of the contraction, k-ranges, pairs of thread blocks, row tiles (needs a GPU)."""
import pytest
import torch

from paper_2603_01399_b200 import binding, synth
from tests.common import gpu_model

pytestmark = pytest.mark.gpu


def _within(y, x, w, scale, res=None):
    """y against the float64 product.  fp32 accumulation: K products are added in K / 16 steps that may truncate, at most
    2^-23 of the sum of magnitudes each, and the sums of up to 8 ranges join; a bf16 output rounds twice (2^-9 each) where a
    residual is added."""
    xd, wd = x.double(), w.double()
    t = (xd @ wd.T) * scale
    mag = (xd.abs() @ wd.abs().T) * scale.abs()
    bound = mag * ((x.shape[1] / 16 + 24) * 2.0 ** -23)
    if res is not None:
        bound = bound + t.abs() * 2.0 ** -8
        t = t + res.double()
    if y.dtype == torch.bfloat16:
        bound = bound + t.abs() * 2.0 ** -8
    assert bool(((y.double() - t).abs() <= bound + 1e-30).all()), ((y.double() - t).abs() - bound).max()


# rows: one tile of digit rows, its edge (64), wide blocks of one and more row tiles; channels: part of a tile, an odd count,
# a tile and a bit, more tiles than SMs; contraction: one block with a tail, ranges, long
SIZES = [(1, 129, 1040), (1, 64, 528), (5, 4096, 4096), (6, 4096, 12288), (15, 1001, 2064), (8, 40, 512), (9, 257, 16), (16, 4096, 4096), (17, 1000, 528), (63, 1001, 4112), (64, 4104, 2064), (64, 20480, 272), (65, 333, 2064), (72, 4104, 2064), (80, 24576, 256), (81, 333, 2064),
         (81, 128, 16), (96, 4096, 4096), (128, 257, 1040), (176, 20480, 272), (193, 512, 4096), (256, 1001, 2048), (257, 4096, 1040), (512, 600, 4112)]


@pytest.mark.parametrize("weights", ["int8", "bf16"])
@pytest.mark.parametrize("m,n,k", SIZES)
def test_linear_forms(m, n, k, weights):
    x = synth.normal_bf16((m, k), 1.0, seed=m + n, device="cuda")
    x[m // 2] *= 2.0 ** 60                     # a row of its own range
    w = synth.normal_bf16((n, k), 0.02, seed=n + k, device="cuda")
    scale = torch.ones(n, dtype=torch.float64, device="cuda")
    q, d = w, None
    if weights == "int8":
        q, d = binding.quasar_quantize(w)
        scale = d.double()
    res = synth.normal_bf16((m, n), 1.0, seed=7, device="cuda")
    _within(binding.quasar_linear(x, q, d, out_f32=True), x, q, scale)
    _within(binding.quasar_linear(x, q, d, residual=res), x, q, scale, res)


@pytest.mark.parametrize("m,n,k", [s for s in SIZES if s[0] <= 256])
def test_w8a8_forms(m, n, k):
    x = synth.normal_bf16((m, k), 1.0, seed=m + n, device="cuda")
    q, d = binding.quasar_quantize(synth.normal_bf16((n, k), 0.02, seed=n + k, device="cuda"))
    codes, dx = binding.quasar_quantize_activations(x, None)
    y, acc = binding.quasar_linear_w8a8(x, None, q, d, out_f32=True, want_acc=True)
    want = (codes.double() @ q.double().T)     # exact: below 2^53
    assert torch.equal(acc.double(), want)
    assert torch.equal(y, want.float() * (d[None, :] * dx[:, None]))


def _batch_against_alone(m, rows, parents=None, tol=1e-2):
    shape, s_max, B = m.shape, 448, 8
    lens = [0, 1, 127, 128, 129, 200, 300, 384]
    kk, vv = synth.kv_prefix(shape, B, s_max, seed=3, device="cuda")
    tokens = synth.uniform_tokens((B, rows), shape.vocab, 5).to(torch.int32)
    block = [max(1, rows - 3 * b) for b in range(B)]

    def run(which):
        kv = binding.KVCache(shape, len(which), s_max, k=kk[:, which].contiguous(), v=vv[:, which].contiguous(),
                             seq_len=torch.tensor([lens[b] for b in which], dtype=torch.int32, device="cuda"))
        buf = binding.VerifyBuffers(m, len(which), rows, tree=parents is not None)
        buf.tokens.copy_(tokens[which])
        if parents is not None:
            buf.parents.copy_(parents[which])
        buf.block_len.copy_(torch.tensor([block[b] for b in which], dtype=torch.int32))
        binding.quasar_verify(m, kv, buf)
        torch.cuda.synchronize()
        assert int(buf.status[0]) == 0
        return buf, kv

    every, kv = run(list(range(B)))
    for b in range(B):
        alone, kv1 = run([b])
        a, e = alone.logits[0, :block[b]].double(), every.logits[b, :block[b]].double()
        assert float((a - e).norm() / a.norm()) <= tol, b
        p = lens[b]
        for x, y in ((kv1.k, kv.k), (kv1.v, kv.v)):
            u, v = x[:, 0, :, p:p + block[b]].double(), y[:, b, :, p:p + block[b]].double()
            assert float((u - v).norm() / u.norm()) <= tol, b
            assert torch.equal(x[:, 0, :, :p], y[:, b, :, :p])


@pytest.mark.parametrize("kind", ["int8", "bf16"])
@pytest.mark.parametrize("name,rows", [("tiny", 10), ("tiny", 11), ("tiny_qknorm", 16), ("tiny_qknorm", 17), ("tiny", 64)])
def test_a_batch_gives_what_its_sequences_give_alone(name, rows, kind):
    """8 x rows block rows take other forms of the linear layers than rows do (fused epilogues up to 64 rows of digits and 128
    otherwise, wide blocks beyond); the attention deals out more pieces than one.  Sums in another order: bf16 roundings,
    1e-2 of the logits, as between the two forms of the pass."""
    _batch_against_alone(gpu_model(synth.SHAPES[name], seed=0, int8=kind == "int8", max_seq=448), rows)


@pytest.mark.parametrize("name,rows", [("tiny", 9), ("tiny_qknorm", 16), ("tiny", 17), ("tiny_qknorm", 64)])
def test_a_w8a8_batch_gives_what_its_sequences_give_alone(name, rows):
    """8 x rows: 72 and 128 rows with the fused epilogues, 136 and 512 without.  A last bit of a norm becomes a quantisation step
    now and then, 1/127 of a row's maximum."""
    _batch_against_alone(gpu_model(synth.SHAPES[name], seed=0, max_seq=448, act_int8=True), rows, tol=2e-2)


@pytest.mark.parametrize("kind", ["int8", "w8a8", "bf16"])
@pytest.mark.parametrize("rows", [8, 9, 17])
def test_a_batch_of_trees_gives_what_its_trees_give_alone(rows, kind):
    """64 rows (digits, fused), 72 (the wide form) and 136 of random trees, each sequence with one of its own."""
    g = torch.Generator().manual_seed(rows)
    parents = torch.tensor([[-1] + [int(torch.randint(0, i, (1,), generator=g)) for i in range(1, rows)] for _ in range(8)], dtype=torch.int32)
    m = gpu_model(synth.SHAPES["tiny_qknorm"], seed=0, int8=kind != "bf16", max_seq=448, act_int8=kind == "w8a8")
    _batch_against_alone(m, rows, parents, 2e-2 if kind == "w8a8" else 1e-2)


@pytest.mark.parametrize("k", [512, 4096])
@pytest.mark.parametrize("m", [1, 6, 7, 8, 64, 65, 80, 81])
def test_a_row_with_a_nan_or_an_infinity_does_not_turn_into_numbers(m, k):
    """NaN: the whole row.  One infinity: that of the sign of the weight it meets, NaN where that is zero (as a sum of IEEE
    products).  The other rows are what they were."""
    n = 300
    x = synth.normal_bf16((m, k), 1.0, seed=m, device="cuda")
    q, d = binding.quasar_quantize(synth.normal_bf16((n, k), 0.02, seed=k, device="cuda"))
    q[::7, k - 3] = 0
    clean = binding.quasar_linear(x, q, d, out_f32=True)
    for value in (float("nan"), float("inf"), -float("inf")):
        bad = x.clone()
        bad[m // 2, k - 3] = value
        y = binding.quasar_linear(bad, q, d, out_f32=True)
        want = clean.clone()
        want[m // 2] = value * q[:, k - 3].float()
        assert torch.equal(torch.nan_to_num(y, nan=12345.0), torch.nan_to_num(want, nan=12345.0)), value


@pytest.mark.parametrize("traced", [False, True])
@pytest.mark.parametrize("rows", [5, 8, 9, 17])
def test_a_nan_on_its_way_through_the_pass_reaches_the_logits(rows, traced):
    """8 x rows block rows (fused and unfused digit forms, the wide form): a NaN in one sequence's cached V leaves that sequence
    without a finite logit and the others as they were; one out of a gate unit does so to all."""
    shape, B, s_max = synth.SHAPES["tiny"], 8, 64
    m = gpu_model(shape, seed=0, max_seq=s_max)
    kk, vv = synth.kv_prefix(shape, B, s_max, seed=3, device="cuda")
    tokens = synth.uniform_tokens((B, rows), shape.vocab, 5).to(torch.int32)

    def run(v):
        kv = binding.KVCache(shape, B, s_max, k=kk.clone(), v=v.clone(), seq_len=torch.full((B,), 40, dtype=torch.int32, device="cuda"))
        buf = binding.VerifyBuffers(m, B, rows)
        buf.tokens.copy_(tokens)
        if traced:
            m.set_trace(torch.empty(m.trace_bytes(B, rows), dtype=torch.uint8, device="cuda"))
        binding.quasar_verify(m, kv, buf)
        torch.cuda.synchronize()
        m.set_trace(None)
        assert int(buf.status[0]) == 0
        return buf.logits

    clean = run(vv)
    assert bool(torch.isfinite(clean).all())
    bad = vv.clone()
    bad[0, 3, 0, 11, 5] = float("nan")
    out = run(bad)
    assert bool(torch.isnan(out[3]).all())
    others = [b for b in range(B) if b != 3]
    assert torch.equal(out[others], clean[others])
    m.tensors["l1.gateup_delta"][3] = float("nan")
    assert bool(torch.isnan(run(vv)).all())


@pytest.mark.parametrize("m", [1, 7, 64, 80])
def test_long_contractions_do_not_wrap(m):
    """Equal elements whose fixed-point form repeats a digit of -128, against weights of 127: from 132,104 products on their sum
    leaves 32 bits.  (Eight k-ranges of 137,500 here.)  An fp32 sum of K / 16 steps, 2^-23 of it each at most."""
    n, k = 40, 1_100_000
    q = torch.full((n, k), 127, dtype=torch.int8, device="cuda")
    d = torch.ones(n, device="cuda")
    for value in (1 + 2.0 ** -5, 1 + 2.0 ** -7):
        x = torch.full((m, k), value, device="cuda").to(torch.bfloat16)
        y = binding.quasar_linear(x, q, d, out_f32=True).double()
        want = value * 127 * k
        assert float((y - want).abs().max()) <= want * (k / 16) * 2.0 ** -23


@pytest.mark.parametrize("k", [2064, 4096])
@pytest.mark.parametrize("m", [1, 6, 7, 16, 64, 65, 80, 81])
def test_what_stands_beside_an_outlier_keeps_its_precision(m, k):
    """An element of 2^14 among normal ones, met by weights of zero: it adds nothing to a product, nor to the bound of one (the
    magnitudes' sum), but a fixed-point form of the row stands against it."""
    n = 600
    x = synth.normal_bf16((m, k), 1.0, seed=m, device="cuda")
    x[:, 3] = 2.0 ** 14
    q, d = binding.quasar_quantize(synth.normal_bf16((n, k), 0.02, seed=k, device="cuda"))
    q[:, 3] = 0
    _within(binding.quasar_linear(x, q, d, out_f32=True), x, q, d.double())


@pytest.mark.parametrize("m", [1, 7, 64, 65])
def test_rows_up_to_the_largest_and_down_to_the_smallest_numbers(m):
    """The powers of two on either side of a row's digits stay normal numbers for every finite bf16 row; a maximum just below a
    power of two has room among the digits."""
    k, n = 1040, 130
    q = torch.zeros((n, k), dtype=torch.int8, device="cuda")
    q[:, 5], q[:, 1039] = 1, -2
    q[7, 6] = 127
    d = torch.ones(n, device="cuda")
    for top in (3.3895313892515355e38, 3.0e38, 255.0, 2.0 ** 31, 2.0 ** -94):
        x = torch.zeros((m, k), device="cuda", dtype=torch.bfloat16)
        x[:, 5], x[:, 1039], x[:, 6] = top, top / 8, -top / 256
        want = (x.double() @ q.double().T).float()
        assert torch.allclose(binding.quasar_linear(x, q, d, out_f32=True), want, rtol=2.0 ** -20, atol=0.0), top


@pytest.mark.parametrize("m,n,k", [(5, 40, 512), (6, 4096, 4096), (16, 1000, 2064), (64, 4096, 4096), (65, 333, 2064), (80, 24576, 256)])
def test_what_a_workspace_holds_does_not_matter(m, n, k):
    x = synth.normal_bf16((m, k), 1.0, seed=m, device="cuda")
    q, d = binding.quasar_quantize(synth.normal_bf16((n, k), 0.02, seed=n, device="cuda"))
    ws = torch.zeros(binding.quasar_linear_workspace_bytes(m, n, k), dtype=torch.uint8, device="cuda")
    want = binding.quasar_linear(x, q, d, workspace=ws, out_f32=True)
    assert torch.equal(binding.quasar_linear(x, q, d, workspace=ws.fill_(255), out_f32=True), want)
    assert torch.equal(binding.quasar_linear(x, q, d, out_f32=True), want)


@pytest.mark.parametrize("room", [0, 600, 512 + 1 * 8260, 512 + 7 * 8260 + 100, 512 + 20 * 8260])
def test_a_workspace_that_holds_some_of_the_rows(room):
    """Behind the reserved 64 KiB: none of the 20 rows of 4 x 2064 digits and a scale (the warp-level kernel then), one, seven, all."""
    m, n, k = 20, 1001, 2064
    x = synth.normal_bf16((m, k), 1.0, seed=1, device="cuda")
    q, d = binding.quasar_quantize(synth.normal_bf16((n, k), 0.02, seed=2, device="cuda"))
    res = synth.normal_bf16((m, n), 1.0, seed=3, device="cuda")
    ws = torch.full((65536 + room + 4096,), 7, dtype=torch.uint8, device="cuda")
    y = binding.quasar_linear(x, q, d, residual=res, workspace=ws[:65536 + room])
    _within(y, x, q, d.double(), res)
    assert bool((ws[65536 + room:] == 7).all())


# rows: one, some, the most of the form and one more; channels: the narrowest tiles of the form (144), last ones that are cut (160,
# 176), wide ones (208, 256); contraction: many turns of the ring, with a remainder; the last two sizes run in tiles of 128
@pytest.mark.parametrize("hidden,ffn", [(4096, 9536), (3600, 11008), (4096, 12288), (4096, 15392), (1024, 18944), (256, 9536), (256, 12288)])
@pytest.mark.parametrize("batch,rows", [(1, 1), (1, 6), (2, 4), (3, 3)])
def test_gateup_on_bf16_weights_in_one_wave_of_wide_tiles(batch, rows, hidden, ffn):
    """Two gate+up tiles on one thread block (SwiGLU in the epilogue; tests/test_forms_rule.py says which sizes run so) against the
    plain layer and SwiGLU behind it, which a trace asks for: the same sums in another order, so the logits agree as the forms of a
    layer do."""
    shape, s_max = synth.ModelShape("wide_ffn", 1, hidden, 4, 2, 64, ffn, 512, False), 128
    m = gpu_model(shape, seed=0, int8=False, max_seq=s_max, gen_device="cuda")
    kk, vv = synth.kv_prefix(shape, batch, s_max, seed=3, device="cuda")
    tokens = synth.uniform_tokens((batch, rows), shape.vocab, 5).to(torch.int32)

    def run(traced):
        kv = binding.KVCache(shape, batch, s_max, k=kk.clone(), v=vv.clone(), seq_len=torch.full((batch,), 40, dtype=torch.int32, device="cuda"))
        buf = binding.VerifyBuffers(m, batch, rows)
        buf.tokens.copy_(tokens)
        if traced:
            m.set_trace(torch.empty(m.trace_bytes(batch, rows), dtype=torch.uint8, device="cuda"))
        binding.quasar_verify(m, kv, buf)
        torch.cuda.synchronize()
        m.set_trace(None)
        assert int(buf.status[0]) == 0
        return buf.logits

    fused, plain = run(False), run(True)
    # a sum's last bit moves a bf16 tensor by 2^-8 of an element now and then; the logits are sums over 256 or more of them
    assert bool(((fused - plain).abs() <= 2.0 ** -6 * plain.pow(2).mean(dim=-1, keepdim=True).sqrt() + 1e-2 * plain.abs()).all())


# rows: the fewest of the wide form, one row tile with several rows a warp, two row tiles, blocks that end early; heads: whole tiles
# of 256 channels, and a last one cut
@pytest.mark.parametrize("heads,kv_heads,dim,norm", [(8, 2, 128, True), (6, 2, 64, False)])
@pytest.mark.parametrize("batch,rows,tree", [(5, 13, False), (2, 40, False), (5, 60, False), (4, 17, True), (8, 24, False)])
def test_wide_qkv_rows_finish_as_those_of_the_layer_and_the_kernel_behind_it(batch, rows, tree, heads, kv_heads, dim, norm):
    """QK-norm, RoPE and cache append where the sums of the k-ranges join, against the two kernels that a trace asks for: the same
    bits.  The FFNs give zeros, so what stands between one layer's q, k and v and the next one's are the same kernels on both sides:
    a q head in the wrong place or with the wrong gain shows in the second layer's cache rows and in the logits.  No other rows of
    the cache are written."""
    shape, s_max = synth.ModelShape("wide_qkv", 2, 2048, heads, kv_heads, dim, 512, 512, norm), 128
    m = gpu_model(shape, seed=0, int8=True, max_seq=s_max, gen_device="cuda")
    for layer in range(2):
        m.tensors[f"l{layer}.gateup_delta"].zero_()
    kk, vv = synth.kv_prefix(shape, batch, s_max, seed=3, device="cuda")
    tokens = synth.uniform_tokens((batch, rows), shape.vocab, 5).to(torch.int32)
    lens = torch.tensor([rows - b % 3 for b in range(batch)], dtype=torch.int32)
    g = torch.Generator().manual_seed(rows)
    parents = torch.tensor([[-1] + [int(torch.randint(0, i, (1,), generator=g)) for i in range(1, rows)] for _ in range(batch)], dtype=torch.int32)

    def run(traced):
        seq = torch.arange(30, 30 + batch, dtype=torch.int32, device="cuda")
        kv = binding.KVCache(shape, batch, s_max, k=kk.clone(), v=vv.clone(), seq_len=seq)
        buf = binding.VerifyBuffers(m, batch, rows, tree=tree)
        buf.tokens.copy_(tokens)
        buf.block_len.copy_(lens)
        if tree:
            buf.parents.copy_(parents)
        if traced:
            m.set_trace(torch.empty(m.trace_bytes(batch, rows), dtype=torch.uint8, device="cuda"))
        before = binding.kernel_launches()
        binding.quasar_verify(m, kv, buf)
        launches = binding.kernel_launches() - before
        torch.cuda.synchronize()
        m.set_trace(None)
        assert int(buf.status[0]) == 0
        return kv, buf.logits, launches

    (kv, logits, launches), (kv_t, logits_t, launches_t) = run(False), run(True)
    assert launches_t - launches == 2 * 2     # a layer's RoPE kernel and its SwiGLU kernel: both forms ran
    assert torch.equal(kv.k, kv_t.k) and torch.equal(kv.v, kv_t.v)
    rows_written = torch.zeros(batch, s_max, dtype=torch.bool)
    for b in range(batch):
        rows_written[b, 30 + b:30 + b + int(lens[b])] = True
        assert torch.equal(logits[b, :int(lens[b])], logits_t[b, :int(lens[b])])
    for new, old in ((kv.k, kk), (kv.v, vv)):   # [layer][sequence][head][position][channel]
        assert torch.equal((new != old).any(dim=-1).any(dim=2).any(dim=0).cpu(), rows_written)


@pytest.mark.parametrize("top", [254.0, 255.0, 128.0, 129.0])
@pytest.mark.parametrize("k", [256, 4096, 12288])
def test_quantiser_at_the_middles_between_codes(top, k):
    """A row whose maximum is 254 / 256 of a power of two has step sizes that put bf16 values on exact middles all along, other
    maxima near them now and then: the codes are those of the rounded quotient everywhere, of the 4-bit groups too."""
    n = 37
    g = torch.Generator().manual_seed(int(top) + k)
    w = (torch.randint(-int(top), int(top) + 1, (n, k), generator=g).float() * 2.0 ** torch.randint(-9, 1, (n, k), generator=g)).to(torch.bfloat16)
    w[:, ::128] = top
    w = w * 2.0 ** -12
    q, d = binding.quasar_quantize(w.cuda())
    delta = w.float().abs().amax(1) / 127.0
    assert torch.equal(d.cpu(), delta)
    assert torch.equal(q.cpu(), torch.round(w.float() / delta[:, None]).to(torch.int8))
    packed, d4 = binding.quasar_quantize_int4(w.cuda())
    groups = w.float().view(n, k // 128, 128)
    delta4 = groups.abs().amax(2) / 7.0
    codes = torch.round(groups / delta4[..., None]).to(torch.int32).view(n, k)
    assert torch.equal(d4.cpu(), delta4)
    assert torch.equal(packed.cpu().to(torch.int32), (codes[:, ::2] & 15) | ((codes[:, 1::2] & 15) << 4))


# rows: one block of 16 and its edges, two launches; channels: part of a tile, an odd count, more tiles than SMs; groups: one, odd, ranges
@pytest.mark.parametrize("m,n,k", [(1, 129, 128), (15, 1001, 384), (16, 4096, 1152), (17, 130, 640), (33, 19077, 256), (48, 515, 2048),
                                   (64, 20480, 384), (65, 300, 896), (5, 1376, 12288)])
def test_w4_forms(m, n, k):
    x = synth.normal_bf16((m, k), 1.0, seed=m + n, device="cuda")
    packed, d = binding.quasar_quantize_int4(synth.normal_bf16((n, k), 0.02, seed=n + k, device="cuda"))
    p = packed.to(torch.int32)
    codes = torch.stack([p & 15, p >> 4], dim=2).view(n, k)
    w = (codes - 16 * (codes > 7)).double() * d.double().repeat_interleave(128, dim=1)
    res = synth.normal_bf16((m, n), 1.0, seed=7, device="cuda")
    one = torch.ones(n, dtype=torch.float64, device="cuda")
    _within(binding.quasar_linear_w4(x, packed, d, out_f32=True), x, w, one)
    _within(binding.quasar_linear_w4(x, packed, d, residual=res), x, w, one, res)


@pytest.mark.parametrize("batch,rows,prefixes", [(50, 1, (0, 40)), (3, 2, (120, 300)), (1, 6, (900, 900)), (60, 3, (0, 260)), (5, 33, (100, 390))])
def test_sequences_of_a_batch_attend_as_they_do_alone(batch, rows, prefixes):
    """Segments of one key tile and of several, whole on one thread block or shared, more sequences than a block keeps the places
    of: the first layer's attention, by the cache rows of the second and the logits, against each sequence in a batch of its own."""
    shape, s_max = synth.SHAPES["tiny_qknorm"], 960
    m = gpu_model(shape, seed=0, max_seq=s_max)
    kk, vv = synth.kv_prefix(shape, batch, s_max, seed=5, device="cuda")
    lens = torch.tensor([prefixes[0] + (prefixes[1] - prefixes[0]) * b // max(1, batch - 1) for b in range(batch)], dtype=torch.int32, device="cuda")
    tokens = synth.uniform_tokens((batch, rows), shape.vocab, 5).to(torch.int32)

    def run(which):
        kv = binding.KVCache(shape, len(which), s_max, k=kk[:, which].contiguous().clone(), v=vv[:, which].contiguous().clone(), seq_len=lens[which].clone())
        buf = binding.VerifyBuffers(m, len(which), rows)
        buf.tokens.copy_(tokens[which])
        binding.quasar_verify(m, kv, buf)
        torch.cuda.synchronize()
        assert int(buf.status[0]) == 0
        return buf.logits, kv.k, kv.v

    logits, kc, vc = run(list(range(batch)))
    for b in list(range(0, batch, 7)) + [batch - 1]:
        one, k1, v1 = run([b])
        assert bool(((logits[b] - one[0]).abs() <= torch.clamp(1e-2 * one[0].abs(), min=2e-2)).all())
        at = slice(int(lens[b]), int(lens[b]) + rows)
        for got, want in ((kc[1, b, :, at], k1[1, 0, :, at]), (vc[1, b, :, at], v1[1, 0, :, at])):   # two roundings of bf16 apart at most, of the rms where small
            floor = want.float().pow(2).mean().sqrt()
            assert bool(((got.float() - want.float()).abs() <= 2.0 ** -6 * torch.maximum(want.float().abs(), floor)).all())
