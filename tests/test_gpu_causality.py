"""Values that are not finite and causality: an inf or NaN at one position reaches the positions that see it and no
others, in the forward pass (through K and V) and in the backward pass (through K, V, Q and dO)."""
import math

import pytest
import torch

from paper_2407_00952_b200 import binding as B

pytestmark = pytest.mark.gpu


def _seen(weight, value, see):
    """sum over j of weight[..., i, j] * value[..., j, :] over the pairs in `see` only: a hidden pair is not a product with 0."""
    prod = weight[..., None] * value[..., None, :, :]
    return torch.where(see[..., None], prod, torch.zeros((), dtype=prod.dtype, device=prod.device)).sum(-2)


def _reference(qkv, o, lse, do, nseq, T, H, dh):
    """Forward of qkv, and backward from the given o and lse, in 64 bits."""
    q, k, v = (t.transpose(1, 2) for t in qkv.double().view(nseq, T, 3, H, dh).unbind(2))
    o, do = (t.double().view(nseq, T, H, dh).transpose(1, 2) for t in (o, do))
    see = torch.ones(T, T, dtype=torch.bool, device="cuda").tril()
    scale = dh ** -0.5
    z = torch.where(see, (q[..., None, :] * k[..., None, :, :]).sum(-1) * scale, -math.inf)
    # the maximum of the visible scores passes over NaN, as fmaxf does; a NaN score makes its row NaN all the same
    m = torch.where(see & ~z.isnan(), z, -math.inf).amax(-1, keepdim=True)
    p = torch.where(see, torch.exp(z - m), 0.0)
    l = p.sum(-1, keepdim=True)
    fwd_o, fwd_lse = _seen(p, v, see) / l, (m + torch.log(l)).squeeze(-1)
    pb = torch.where(see, torch.exp(z - lse.double()[..., None]), 0.0)
    dp = (do[..., None, :] * v[..., None, :, :]).sum(-1)
    ds = torch.where(see, pb * (dp - (o * do).sum(-1, keepdim=True)) * scale, 0.0)
    dq = _seen(ds, k, see)
    dk, dv = (_seen(w.transpose(-1, -2), x, see.T) for w, x in ((ds, q), (pb, do)))
    rows = lambda t: t.transpose(1, 2).reshape(nseq * T, -1)  # noqa: E731
    return rows(fwd_o), fwd_lse, torch.stack([t.transpose(1, 2) for t in (dq, dk, dv)], 2).reshape(nseq * T, 3 * H * dh)


def _same(got, ref, tol):
    got = got.double()
    assert torch.equal(got.isnan(), ref.isnan())
    assert torch.equal(got.isposinf(), ref.isposinf()) and torch.equal(got.isneginf(), ref.isneginf())
    fine = ref.isfinite()
    assert bool(fine.any()) and float((got - ref)[fine].norm()) <= tol * float(ref[fine].norm())


@pytest.mark.parametrize("where", ["q", "k", "v", "do"])
@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("T,dh", [(70, 24), (64, 40), (33, 5), (9, 128), (100, 64)])
@pytest.mark.parametrize("dtype,use_tc", [(torch.float32, False), (torch.bfloat16, False), (torch.bfloat16, True)])
def test_non_finite_values_reach_what_sees_them_only(T, dh, dtype, use_tc, value, where):
    nseq, H = 2, 2
    d = H * dh
    g = torch.Generator(device="cuda").manual_seed(T + dh)
    qkv = torch.randn(nseq * T, 3 * d, device="cuda", generator=g).to(dtype)
    do = torch.randn(nseq * T, d, device="cuda", generator=g).to(dtype)
    o, lse = B.attention_fwd(qkv, nseq, T, H, use_tc)
    # in the first sequence, first head: one position in the middle and the last one; the rest stays as it was
    for pos in (T // 2, T - 1):
        if where == "do":
            do[pos, 1] = value
        else:
            qkv[pos, "qkv".index(where) * d + 1] = value
    ref = _reference(qkv, o, lse, do, nseq, T, H, dh)
    tol = 1e-5 if dtype == torch.float32 else 1e-2
    if where != "do":
        for got, want in zip(B.attention_fwd(qkv, nseq, T, H, use_tc), ref):
            _same(got, want, tol)
    _same(B.attention_bwd(qkv, o, lse, do, nseq, T, H, use_tc), ref[2], tol)
    assert B.library_status() == 0


@pytest.mark.parametrize("where", ["q", "k", "v", "do"])
@pytest.mark.parametrize("value", [math.inf, math.nan])
@pytest.mark.parametrize("nseq,T,H", [(2, 192, 2), (40, 320, 2)])
def test_non_finite_values_at_odd_multiples_of_64(nseq, T, H, value, where):
    """Width 64, backward, both launch forms: lengths whose last tile of 128 rows is half a tile."""
    _check_backward_in_tiles_of_128(nseq, T, H, value, where)


@pytest.mark.parametrize("where", ["q", "k", "v", "do"])
@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("nseq,T,H", [(2, 200, 2), (80, 200, 2), (80, 70, 2)])
def test_non_finite_values_in_tiles_of_128(nseq, T, H, value, where):
    """Width 64 off the tile sizes, as the kernels with tiles of 128 rows take it: both gradients in one launch (with the
    forward pass in tiles of 64), a launch for each, sequences of one tile."""
    qkv, ref = _check_backward_in_tiles_of_128(nseq, T, H, value, where)
    if where != "do":
        o, lse = B.attention_fwd(qkv, nseq, T, H)
        _same(o[:2 * T], ref[0], 1e-2)
        _same(lse[:2], ref[1], 1e-2)
        assert B.library_status() == 0


def _check_backward_in_tiles_of_128(nseq, T, H, value, where):
    """Bad values in the first and the last tile of the first sequence's first head; the sequences behind it as they were."""
    dh = 64
    d = H * dh
    g = torch.Generator(device="cuda").manual_seed(nseq + T + H)
    qkv = torch.randn(nseq * T, 3 * d, device="cuda", generator=g).bfloat16()
    do = torch.randn(nseq * T, d, device="cuda", generator=g).bfloat16()
    o, lse = B.attention_fwd(qkv, nseq, T, H)
    before = B.attention_bwd(qkv, o, lse, do, nseq, T, H)
    for pos in (T // 3, T - 1):
        if where == "do":
            do[pos, 1] = value
        else:
            qkv[pos, "qkv".index(where) * d + 1] = value
    n = 2                                                      # the reference takes dh times the pairs in memory
    ref = _reference(qkv[:n * T], o[:n * T], lse[:n], do[:n * T], n, T, H, dh)
    got = B.attention_bwd(qkv, o, lse, do, nseq, T, H)
    _same(got[:n * T], ref[2], 1e-2)
    assert torch.equal(got[T:], before[T:])
    assert B.library_status() == 0
    return qkv, ref
