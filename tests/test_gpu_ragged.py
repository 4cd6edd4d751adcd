"""Shapes off the tile sizes of the tensor-core kernels: they run on tensor cores too, with the precision of the
plain-FMA kernels that are the other way to run them."""
import numpy as np
import pytest
import torch

import harness
from paper_2407_00952_b200 import binding as B
from paper_2407_00952_b200 import synth
from test_gpu_parity import TOL_FP32, check_three_calls

pytestmark = pytest.mark.gpu


def _norm_err(got, ref):
    return float((got.double() - ref).norm() / ref.norm().clamp_min(1e-300))


def _attention64(qkv, do, nseq, T, H, dh):
    q, k, v = (t.transpose(1, 2).contiguous().requires_grad_() for t in qkv.double().view(nseq, T, 3, H, dh).unbind(2))
    z = (q @ k.transpose(-1, -2) * dh ** -0.5).masked_fill(~torch.ones(T, T, dtype=torch.bool, device="cuda").tril(), -np.inf)
    o = torch.softmax(z, -1) @ v
    o.backward(do.double().view(nseq, T, H, dh).transpose(1, 2))
    grads = torch.stack([t.grad.transpose(1, 2) for t in (q, k, v)], 2)
    return (o.detach().transpose(1, 2).reshape(nseq * T, H * dh), torch.logsumexp(z.detach(), -1),
            grads.reshape(nseq * T, 3 * H * dh))


@pytest.mark.parametrize("T,dh", [(1, 64), (2, 8), (31, 32), (63, 24), (64, 32), (65, 64), (128, 96), (129, 128), (200, 40),
                                  (333, 64), (257, 104), (191, 16)])
def test_attention_any_length_and_width(T, dh):
    """Against 64 bits: both forms within the rounding of their bf16 outputs (half a unit, 2^-9 on average) and the
    tensor-core form no further off than the plain-FMA kernels (fp32 probabilities); 2 % more is allowed for another order
    of the sums."""
    nseq, H = 3, 2
    d = H * dh
    g = torch.Generator(device="cuda").manual_seed(100 * T + dh)
    qkv = (1.5 * torch.randn(nseq * T, 3 * d, device="cuda", generator=g)).bfloat16()
    do = torch.randn(nseq * T, d, device="cuda", generator=g).bfloat16()
    ref = _attention64(qkv, do, nseq, T, H, dh)
    errs = []
    for tc in (True, False):
        o, lse = B.attention_fwd(qkv, nseq, T, H, use_tensor_cores=tc)
        dqkv = B.attention_bwd(qkv, o, lse, do, nseq, T, H, use_tensor_cores=tc)
        errs.append([_norm_err(a, r) for a, r in zip((o, lse, dqkv), ref)])
    assert B.library_status() == 0
    # lse is an fp32 result: no further off either, up to one rounding of the result (few values at the short lengths)
    for got, plain, bound, most in zip(*errs, (2e-6, 2.0 ** -24, 2e-6), (4e-3, 1e-6, 4e-3)):
        assert got <= 1.02 * plain + bound and max(got, plain) <= most, errs
    static = B.attention_bwd_static(qkv, o, lse, do, nseq, T, H)
    assert torch.equal(static, B.attention_bwd(qkv, o, lse, do, nseq, T, H))


@pytest.mark.parametrize("nseq,T,H", [(1, 129, 1), (40, 65, 4), (150, 70, 1), (2, 127, 70), (3, 191, 2), (2, 193, 3), (1, 257, 5), (5, 333, 12),
                                      (3, 321, 60), (1, 1025, 2), (30, 161, 12)])
def test_attention_of_any_length_in_tiles_of_128(nseq, T, H):
    """Edges of the 128-row tiles, of their 64-row halves and 32-key steps, one and several units of work per CTA, width 64:
    the bounds of test_attention_any_length_and_width, and the same bits from run to run."""
    dh = 64
    g = torch.Generator(device="cuda").manual_seed(nseq * T + H)
    qkv = (1.5 * torch.randn(nseq * T, 3 * H * dh, device="cuda", generator=g)).bfloat16()
    do = torch.randn(nseq * T, H * dh, device="cuda", generator=g).bfloat16()
    o, lse = B.attention_fwd(qkv, nseq, T, H)
    out = (o, lse, B.attention_bwd(qkv, o, lse, do, nseq, T, H))
    plain_o, plain_lse = B.attention_fwd(qkv, nseq, T, H, use_tensor_cores=False)
    plain = (plain_o, plain_lse, B.attention_bwd(qkv, plain_o, plain_lse, do, nseq, T, H, use_tensor_cores=False))
    assert B.library_status() == 0
    for got, other, ref, bound, most in zip(out, plain, _attention64(qkv, do, nseq, T, H, dh), (2e-6, 2.0 ** -24, 2e-6), (4e-3, 1e-6, 4e-3)):
        assert _norm_err(got, ref) <= min(1.02 * _norm_err(other, ref) + bound, most)
    again = B.attention_fwd(qkv, nseq, T, H)
    assert torch.equal(o, again[0]) and torch.equal(lse, again[1]) and torch.equal(out[2], B.attention_bwd(qkv, o, lse, do, nseq, T, H))


@pytest.mark.parametrize("nseq,T,H", [(64, 64, 16), (26, 192, 8), (8, 64, 64), (2, 192, 8)])
def test_attention_forward_of_short_whole_tiles(nseq, T, H):
    """One to three tiles per sequence, more and fewer blocks than three per SM, width 64: within the rounding of the
    probabilities and the output to bf16 (2^-8 each)."""
    dh = 64
    g = torch.Generator(device="cuda").manual_seed(nseq + T)
    qkv = torch.randn(nseq * T, 3 * H * dh, device="cuda", generator=g).bfloat16()
    do = torch.randn(nseq * T, H * dh, device="cuda", generator=g).bfloat16()
    o, lse = B.attention_fwd(qkv, nseq, T, H)
    dqkv = B.attention_bwd(qkv, o, lse, do, nseq, T, H)
    ref = _attention64(qkv, do, nseq, T, H, dh)
    assert [_norm_err(a, r) <= b for a, r, b in zip((o, lse, dqkv), ref, (2 * 2.0 ** -8, 1e-6, 3 * 2.0 ** -8))] == [True] * 3


@pytest.mark.parametrize("T", [1, 2, 5, 6, 8, 9, 10, 11, 16, 17])
@pytest.mark.parametrize("dh", [5, 32, 64, 128])
@pytest.mark.parametrize("nseq,H", [(2, 3), (150, 4)])
def test_attention_of_short_sequences(T, dh, nseq, H):
    """Both sides of the lengths and head counts at which short sequences change kernels (tiles, a warp per row, tensor
    cores), fp32 and bf16.  fp32: about as many roundings of random sign as terms in a score and in a row's sum, taken four
    times; bf16: the rounding of the output."""
    g = torch.Generator(device="cuda").manual_seed(T * dh + nseq)
    for dtype, bounds in ((torch.float32, [4 * (T + dh) ** 0.5 * 2.0 ** -24] * 3), (torch.bfloat16, (4e-3, 1e-6, 4e-3))):
        qkv = torch.randn(nseq * T, 3 * H * dh, device="cuda", generator=g).to(dtype)
        do = torch.randn(nseq * T, H * dh, device="cuda", generator=g).to(dtype)
        o, lse = B.attention_fwd(qkv, nseq, T, H)
        dqkv = B.attention_bwd(qkv, o, lse, do, nseq, T, H)
        errs = [_norm_err(a, r) for a, r in zip((o, lse, dqkv), _attention64(qkv, do, nseq, T, H, dh))]
        assert all(e <= b for e, b in zip(errs, bounds)), (dtype, errs)
        assert torch.equal(dqkv, B.attention_bwd_static(qkv, o, lse, do, nseq, T, H))
    assert B.library_status() == 0


def test_attention_ragged_writes_inside_its_rows_only():
    nseq, T, H, dh = 2, 77, 2, 24
    d, guard = H * dh, 64
    qkv = torch.randn(nseq * T, 3 * d, device="cuda").bfloat16()
    do = torch.randn(nseq * T, d, device="cuda").bfloat16()
    o, lse = B.attention_fwd(qkv, nseq, T, H)
    buf = torch.full((nseq * T + 2 * guard, 3 * d), 7.0, device="cuda", dtype=torch.bfloat16)
    inner = buf[guard:guard + nseq * T]
    B.attention_bwd_static(qkv, o, lse, do, nseq, T, H, dqkv=inner)
    assert bool((buf[:guard] == 7).all()) and bool((buf[guard + nseq * T:] == 7).all())
    assert torch.equal(inner, B.attention_bwd(qkv, o, lse, do, nseq, T, H))


@pytest.mark.parametrize("M,K,N", [(1, 8, 8), (5, 72, 264), (127, 64, 72), (129, 200, 256), (255, 768, 1000), (257, 128, 520),
                                   (1000, 136, 256), (300, 1000, 8),
                                   # few tiles: every split of the contraction, both tile widths, tails of each
                                   (128, 4096, 64), (512, 1024, 64), (256, 512, 64), (512, 4096, 1024), (300, 584, 1000),
                                   (1024, 1024, 1024), (512, 1024, 3072), (2000, 1032, 1000),
                                   # as many tiles as clusters of four or eight would have SMs, and one more than fit
                                   (384, 768, 768), (384, 584, 768), (1920, 4096, 64), (2048, 4096, 64),
                                   # many tiles: CTA pairs (whole tiles, a ragged last one, one whose second CTA has no
                                   # row, half a tile) and one CTA per tile (whole and ragged)
                                   (2048, 768, 3072), (1665, 768, 3072), (4001, 1000, 4096), (2100, 264, 2048), (2176, 768, 3072),
                                   (1152, 1024, 4096), (1100, 1000, 4096)])
@pytest.mark.parametrize("epilogue", [B.EPI_BIAS, B.EPI_BIAS_GELU, B.EPI_BIAS_RESID, B.EPI_MUL_GELUGRAD])
def test_linear_any_row_count_and_depth(M, K, N, epilogue):
    """Against 64 bits: both kernels within the rounding of a bf16 result (2^-8 at most; for GELU also that of the stored
    pre-activation), and the tensor-core one no further off than plain FMA (the products of bf16 values are exact in both and
    both round to bf16 once, so the errors agree to a few per mille); rows past M stay untouched.  With 3e5 results and
    more, the two orders of the sums round a few of them differently: equal bits would mean one kernel ran twice."""
    g = torch.Generator(device="cuda").manual_seed(M + K + N)
    mk = lambda *s, sc=1.0: (torch.randn(*s, device="cuda", generator=g) * sc).bfloat16()  # noqa: E731
    x, W, bias, r = mk(M, K), mk(N, K, sc=K ** -0.5), mk(N), mk(M, N, sc=2.0)
    acc = x.double() @ W.double().T
    z = (acc + bias.double())
    gelu = lambda t: torch.nn.functional.gelu(t, approximate="tanh")  # noqa: E731
    if epilogue == B.EPI_MUL_GELUGRAD:
        t = r.double().requires_grad_()
        gelu(t).sum().backward()
        ref = acc * t.grad
    else:
        ref = {B.EPI_BIAS: z, B.EPI_BIAS_GELU: gelu(z), B.EPI_BIAS_RESID: z + r.double()}[epilogue]
    errs, results = [], []
    for tc in (True, False):
        buf = torch.full((M + 160, N), 7.0, device="cuda", dtype=torch.bfloat16)
        zbuf = torch.full((M + 160, N), 7.0, device="cuda", dtype=torch.bfloat16)
        B.linear(x, W, None if epilogue == B.EPI_MUL_GELUGRAD else bias, epilogue, r=r, y=buf[:M], z=zbuf[:M], use_tensor_cores=tc)
        assert bool((buf[M:] == 7).all()) and bool((zbuf[M:] == 7).all())
        errs.append([_norm_err(buf[:M], ref)] + ([_norm_err(zbuf[:M], z)] if epilogue == B.EPI_BIAS_GELU else []))
        results.append(buf)
    most = 2.0 ** -8 * (2 if epilogue == B.EPI_BIAS_GELU else 1)
    for got, plain in zip(*errs):
        # tanh.approx of whole tiles: 2^-11 of the value, far below the rounding of the result
        assert got <= 1.02 * plain + 2e-5 and max(got, plain) <= most, errs
    assert M * N < 300_000 or K < 200 or not torch.equal(*results)


@pytest.mark.parametrize("epilogue", [B.EPI_BIAS_GELU, B.EPI_MUL_GELUGRAD])
def test_gelu_off_the_tile_sizes_for_every_pre_activation(epilogue):
    """All bf16 pre-activations up to 1e4 through a layer whose product is exact: the result is the 64-bit value rounded to
    bf16, but for fp32 errors before that rounding.  They are relative to s = sigmoid(2u): three roundings of the exponent,
    2^-24 of 2u each, 2^-22 of the exponential, eight roundings of the rest; the derivative is a sum of s and
    z s (1 - s) d2u/dz, which cancels near z = -0.75.  No more values are misrounded than in plain FMA."""
    bits = torch.arange(65536, dtype=torch.int32, device="cuda").to(torch.int16).view(torch.bfloat16)
    z = bits[bits.isfinite() & (bits.abs() <= 1e4)]
    M, K, N = z.numel(), 8, 8
    x, W = (torch.zeros(n, K, device="cuda", dtype=torch.bfloat16) for n in (M, N))
    W[:, 0] = 1
    z64 = z.double().requires_grad_()
    gelu = torch.nn.functional.gelu(z64, approximate="tanh")
    # the exact product 0.5 z (1 + tanh u) = z / (1 + exp(-2u)); torch's own form cancels in 64 bits far out
    u2 = 2 * (2 / np.pi) ** 0.5 * (z64 + 0.044715 * z64 ** 3)
    s = torch.sigmoid(u2)
    assert float((gelu - z64 * s).detach().abs().max()) < 1e-11
    rel = (3 * u2.detach().abs() + 12) * 2.0 ** -24
    if epilogue == B.EPI_BIAS_GELU:
        ref = (z64 * s).detach()
        slack = rel * ref.abs()
        x[:, 0] = z
    else:
        ds = s * torch.sigmoid(-u2) * 2 * (2 / np.pi) ** 0.5 * (1 + 0.134145 * z64 ** 2)
        ref = (s + z64 * ds).detach()
        slack = rel * (s + 2 * (z64 * ds).abs()).detach()
        x[:, 0] = 1
    r = z[:, None].expand(M, N).contiguous()
    wrong = []
    for tc in (True, False):
        out = B.linear(x, W, None, epilogue, r=r, use_tensor_cores=tc)
        y = (out[0] if epilogue == B.EPI_BIAS_GELU else out)[:, 3].double()
        wrong.append(int((y != ref.bfloat16().double()).sum()))
        if tc:
            slack = slack + (1 + z.double().abs()) ** 3 * 2.0 ** -126      # exponentials below 2^-126 count as 0
            ok = ((y >= (ref - slack).bfloat16().double()) & (y <= (ref + slack).bfloat16().double()))
            assert bool(ok.all()), (z[~ok], y[~ok], ref[~ok])
    assert wrong[0] <= wrong[1], wrong


@pytest.mark.parametrize("M,n_in,n_out,r,G", [(1, 64, 72, 4, 1), (77, 200, 136, 6, 1), (129, 768, 256, 1, 1), (300, 136, 768, 40, 1),
                                              (512, 200, 1000, 8, 2), (640, 72, 72, 64, 5),
                                              (512, 1024, 1024, 4, 2), (256, 4096, 512, 16, 1), (1024, 1024, 1024, 40, 4)])
def test_lora_linear_any_size(M, n_in, n_out, r, G):
    """Forward and backward against 64 bits: within two bf16 roundings (the rank-r projection and the result), and no
    further off than the plain-FMA kernels."""
    g = torch.Generator(device="cuda").manual_seed(M + n_in)
    x = torch.randn(M, n_in, device="cuda", generator=g).bfloat16()
    W = (torch.randn(n_out, n_in, device="cuda", generator=g) * n_in ** -0.5).bfloat16()
    dy = (torch.randn(M, n_out, device="cuda", generator=g) * n_out ** -0.5).bfloat16()
    A = torch.randn(G, r, n_in, device="cuda", generator=g, dtype=torch.float32) * n_in ** -0.5
    Bm = torch.randn(G, n_out, r, device="cuda", generator=g, dtype=torch.float32) * r ** -0.5
    s = 16.0 / r
    xg, dyg, A64, B64 = x.double().view(G, -1, n_in), dy.double().view(G, -1, n_out), A.double(), Bm.double()
    h, dh = xg @ A64.transpose(1, 2), s * dyg @ B64
    ref = ((x.double() @ W.double().T + s * (h @ B64.transpose(1, 2)).reshape(M, n_out)), (dy.double() @ W.double() + (dh @ A64).reshape(M, n_in)),
           dh.transpose(1, 2) @ xg, s * dyg.transpose(1, 2) @ h)
    errs = []
    for tc in (True, False):
        y = B.lora_linear_fwd(x, W, None, A, Bm, 16.0, use_tensor_cores=tc)
        got = (y,) + B.lora_linear_bwd(x, B.transpose(W), dy, A, Bm, 16.0, use_tensor_cores=tc)
        errs.append([_norm_err(a, b) for a, b in zip(got, ref)])
    assert B.library_status() == 0
    for got, plain in zip(*errs):
        assert got <= 1.02 * plain + 2e-5 and max(got, plain) <= 2 * 2.0 ** -8, errs


@pytest.mark.parametrize("M,K,N", [(1, 8, 8), (33, 72, 40), (65, 136, 200), (512, 1024, 128), (31, 64, 1000), (700, 200, 1000),
                                   (1600, 40, 1608)])
def test_linear_fp32_any_size(M, K, N):
    """Both tile sizes and the unaligned form: every element within the bound of a K-term fp32 sum in any order,
    (K + 2) 2^-24 sum |x w|; rows past M stay untouched."""
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x, W = (torch.randn(*s, device="cuda", generator=g, dtype=torch.float32) for s in ((M, K), (N, K)))
    bias, r = (torch.randn(*s, device="cuda", generator=g, dtype=torch.float32) for s in ((N,), (M, N)))
    ref = x.double() @ W.double().T + bias.double() + r.double()
    bound = (K + 2) * 2.0 ** -24 * (x.double().abs() @ W.double().abs().T + bias.double().abs() + r.double().abs())
    shifted = torch.empty(M * K + 1, device="cuda", dtype=torch.float32)[1:].view(M, K).copy_(x)
    for xin in (x, shifted):
        buf = torch.full((M + 64, N), 7.0, device="cuda", dtype=torch.float32)
        B.linear(xin, W, bias, B.EPI_BIAS_RESID, r=r, y=buf[:M])
        assert bool((buf[M:] == 7).all()) and bool(((buf[:M].double() - ref).abs() <= bound).all())


@pytest.mark.parametrize("M,n_in,n_out,r,G", [(15, 1024, 1032, 8, 1), (17, 1000, 2304, 9, 1), (33, 3080, 40, 7, 1), (100, 4104, 64, 8, 1),
                                              (2048, 2048, 2056, 12, 2), (4096, 256, 4096, 16, 1), (4097, 1024, 256, 8, 1), (256, 1024, 1024, 33, 1)])
def test_rank_projections_of_every_shape(M, n_in, n_out, r, G):
    """Rows and columns around the tiles and slabs of the rank-r projections, one to four slabs and more than they take, ranks
    around their column tiles, and the row counts at which they hand over to the linear layers' kernels."""
    test_lora_linear_any_size(M, n_in, n_out, r, G)


@pytest.mark.parametrize("T,H,dh", [(64, 4, 32), (100, 4, 64), (37, 3, 40), (200, 2, 128), (65, 2, 96), (50, 2, 5)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_plain_attention_backward_does_not_depend_on_the_batch(T, H, dh, dtype):
    """Few blocks take both gradients in one launch, many a kernel for each: a sequence's gradients are the same bits."""
    few, many = 1, 200
    g = torch.Generator(device="cuda").manual_seed(T + dh)
    qkv = torch.randn(many * T, 3 * H * dh, device="cuda", generator=g).to(dtype)
    do = torch.randn(many * T, H * dh, device="cuda", generator=g).to(dtype)
    o, lse = B.attention_fwd(qkv, many, T, H, use_tensor_cores=False)
    n = few * T
    part = B.attention_bwd(qkv[:n], o[:n].contiguous(), lse[:few].contiguous(), do[:n], few, T, H, use_tensor_cores=False)
    assert torch.equal(part, B.attention_bwd(qkv, o, lse, do, many, T, H, use_tensor_cores=False)[:n])


@pytest.mark.parametrize("M,K,N", [(1, 8, 8), (512, 128, 64), (512, 512, 128), (100, 520, 128), (77, 1000, 40), (512, 128, 384), (1200, 72, 1000)])
def test_linear_fp32_tiles(M, K, N):
    """Few to many tiles, with the contraction over one, four, eight and sixteen thread groups: roundings of random sign, one
    per term of the longest sum, taken four times."""
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x, W = (torch.randn(n, K, device="cuda", generator=g, dtype=torch.float32) for n in (M, N))
    buf = torch.full((M + 16, N), 7.0, device="cuda", dtype=torch.float32)
    B.linear(x, W, None, y=buf[:M])
    assert bool((buf[M:] == 7).all())
    assert _norm_err(buf[:M], x.double() @ W.double().T) <= 4 * K ** 0.5 * 2.0 ** -24


@pytest.mark.parametrize("M,K,N", [(1000, 2304, 768), (999, 4096, 1000), (1700, 1032, 2952), (1665, 768, 2304)])
@pytest.mark.parametrize("epilogue", [B.EPI_BIAS, B.EPI_BIAS_GELU, B.EPI_BIAS_RESID, B.EPI_MUL_GELUGRAD])
def test_linear_tiles_of_128_columns(M, K, N, epilogue):
    """Clusters of two and CTA pairs on tiles of 128 columns, whole and ragged, one and several tiles per pair."""
    test_linear_any_row_count_and_depth(M, K, N, epilogue)


@pytest.mark.parametrize("name", sorted(harness.RAGGED_ROUNDS))
def test_bf16_rounds_off_the_tile_sizes(name):
    """Whole passes whose rows end inside a tile of every kernel: norm and projection in one launch, adapter gradients of all
    layers of a side from planes whose last block is partial, attention, linear layers; the general bounds, which
    test_storage_noise.py shows to hold for these cases."""
    w, _, bound = harness.qk_case(name)
    assert bound is None
    eng = check_three_calls(w, harness.TOL_BF16)
    assert eng.device_status() == 0


def test_fp32_round_off_the_tile_sizes():
    check_three_calls(synth.scaled(synth.WORKLOADS[1], n_layer=4, cut=2, n_clients=1, counts=(7,), batch_per_client=3, seq=37, max_seq=37), TOL_FP32)
