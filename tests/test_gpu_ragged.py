"""Shapes off the tile sizes of the tensor-core kernels: they run on tensor cores too, with the precision of the
plain-FMA kernels that are the other way to run them."""
import numpy as np
import pytest
import torch

from paper_2407_00952_b200 import binding as B

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
    """Against 64 bits: no further off than the plain-FMA kernels (fp32 probabilities), whose error is that of the
    bf16 output; 2 % more is allowed for another order of the sums.  Rows around the tensors stay untouched."""
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
    # lse is an fp32 result: half a unit in its last place, and as much again for every 16-deep step of a score's
    # accumulation, which the tensor core rounds towards zero (at most one unit of the partial sum per step)
    lse_bound = (1 + (dh + 15) // 16) * 2.0 ** -24
    for got, plain, bound in zip(*errs, (2e-6, lse_bound, 2e-6)):
        assert got <= 1.02 * plain + bound, errs
    static = B.attention_bwd_static(qkv, o, lse, do, nseq, T, H)
    assert torch.equal(static, B.attention_bwd(qkv, o, lse, do, nseq, T, H))


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
