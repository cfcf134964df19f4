"""top-k / top-p selection at the edges of its one-pass kernel: slices of 8192 bf16 or 4096 fp32 logits, rows that start
on no 16-byte boundary, candidate lists and bins at their limits, first slices that say nothing about the rest."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_16994_b200 import binding
from .parity import PROB_TOL

pytestmark = pytest.mark.gpu
BF, F32 = torch.bfloat16, torch.float32


def check(z, trunc, T=1.0):
    probs, stats = binding.tree_probs(z, 0, temperature=T, **trunc)
    B, N, V = z.shape
    zb = z.contiguous().cpu()
    bits = zb.view(torch.int16).numpy().view(np.uint16) if z.dtype == BF else zb.numpy()
    inp = oracle.TreeInputs(bits, bits, np.array([-1] + [0] * (N - 1), np.int32), np.zeros((B, N), np.int32),
                            np.zeros((B, N), np.float32), np.zeros((B, N), np.float32), temperature=T,
                            top_k=trunc.get("top_k", 0), top_p=trunc.get("top_p", 1.0))
    rp, rs, _ = oracle.tree_probs(inp, 0)
    sure = rs[..., 5] >= 1e-6                      # rows whose nucleus boundary is not within 1e-6 of top_p
    assert sure.any()
    st = stats.cpu().numpy()
    assert np.abs(probs.cpu().numpy() - rp)[sure].max() < PROB_TOL
    np.testing.assert_array_equal(st[..., 2][sure], rs[..., 2][sure])                          # kept count
    np.testing.assert_array_equal(st[..., 5][sure], rs[..., 6][sure].astype(np.float32))       # threshold logit


def rows(V, dtype, scale=3.0):
    g = torch.Generator(device="cuda").manual_seed(11)
    z = (torch.randn((2, 3, V), generator=g, device="cuda") * scale).to(dtype)
    z[0, 0, : V // 2] = z[0, 0, V // 2: 2 * (V // 2)]          # exact ties everywhere in one row
    z[1, 1, 5], z[1, 1, 6] = -0.0, 0.0
    return z


@pytest.mark.parametrize("V", [7, 4097, 8191, 8192, 8193, 24577])
@pytest.mark.parametrize("dtype", [BF, F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("trunc", [dict(top_k=5), dict(top_p=0.9), dict(top_p=0.99)], ids=["k5", "p90", "p99"])
def test_slice_edges(V, dtype, trunc):
    check(rows(V, dtype), trunc)


@pytest.mark.parametrize("V,dtype,scale,trunc", [
    (40000, BF, 3.0, dict(top_k=1024)), (40000, BF, 3.0, dict(top_k=1025)),      # the last k a first slice bounds, and one more
    (40000, F32, 3.0, dict(top_k=256)), (40000, F32, 3.0, dict(top_k=257)),
    (40000, F32, 3.0, dict(top_p=0.97)),                                        # more candidates than the list of keys holds
    (40000, BF, 300.0, dict(top_k=40)), (40000, BF, 300.0, dict(top_p=0.9)),     # values beyond the bins
    (40000, BF, 0.2, dict(top_p=0.95)),                                         # a nucleus that reaches below zero
    (131072, BF, 1.0, dict(top_p=0.999)),                                       # almost all of the row, counted densely
])
def test_limits(V, dtype, scale, trunc):
    check(rows(V, dtype, scale), trunc)


@pytest.mark.parametrize("dtype", [BF, F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("trunc", [dict(top_k=60), dict(top_p=0.95), dict(top_k=200, top_p=0.9)], ids=["k60", "p95", "k200p90"])
@pytest.mark.parametrize("order", ["descending", "ascending", "minus_inf_first"])
def test_first_slice_unlike_the_rest(dtype, trunc, order):
    V = 50003
    g = torch.Generator(device="cuda").manual_seed(3)
    z = (torch.randn((1, 2, V), generator=g, device="cuda") * 2.5).to(dtype)
    if order == "minus_inf_first":
        z[..., :9000] = -float("inf")
    else:
        z = torch.sort(z.float(), dim=-1, descending=order == "descending").values.to(dtype)
    check(z, trunc, T=0.7)


@pytest.mark.parametrize("V", [20000, 150001], ids=["3_slices", "19_slices"])
@pytest.mark.parametrize("shift,scale,p", [(-40.0, 3.0, 0.95),      # no positive logit: the first slice is counted again
                                           (0.0, 0.5, 0.99),        # a nucleus that reaches far below zero
                                           (1.5, 1.0, 0.9),         # a cut next to the bins that share values
                                           (12.0, 3.0, 0.99), (12.0, 3.0, 0.5)])
def test_bounds_from_the_first_slices(V, shift, scale, p):
    g = torch.Generator(device="cuda").manual_seed(5)
    z = (torch.randn((1, 3, V), generator=g, device="cuda") * scale + shift).to(BF)
    z[0, 1, 8192:] -= 6.0                          # all the mass in the first slice
    z[0, 2, :8192] -= 6.0                          # ... and next to none
    check(z, dict(top_p=p))


def test_a_value_beyond_the_bins_late_in_the_row():
    z = rows(40000, BF)
    z[0, 0, 30000], z[1, 2, 39999], z[1, 0, 100] = 600.0, 511.0, -700.0
    check(z, dict(top_p=0.95), T=200.0)


# temperatures so low that z log2(e) / T leaves the range of the rows' references (1e9): the mass the pass has summed is not known then
@pytest.mark.parametrize("V", [50, 8193, 40000])
@pytest.mark.parametrize("dtype", [BF, F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("shift", [0.0, -40.0])
@pytest.mark.parametrize("trunc", [dict(top_k=5), dict(top_p=0.95), dict(top_k=5, top_p=0.95)], ids=["k5", "p95", "k5p95"])
def test_cuts_beyond_the_range_of_references(V, dtype, shift, trunc):
    z = rows(V, dtype)
    z = (z.float() + shift).to(dtype)
    for T in (1e-7, 1e-9, 1e-12):
        _, stats = binding.tree_probs(z, 0, temperature=T, want_probs=False, **trunc)
        st, zd = stats.cpu().numpy(), z.float().cpu().numpy()
        # a step between neighbouring logits is 13 octaves at least: the nucleus is the maximum and its ties
        if "top_p" in trunc:
            cut = zd.max(-1)
        else:
            cut = -np.sort(-zd, axis=-1)[..., trunc["top_k"] - 1]
        np.testing.assert_array_equal(st[..., 5], cut)
        np.testing.assert_array_equal(st[..., 2], (zd >= cut[..., None]).sum(-1))


# Masked vocabularies: fewer ordinary tokens than top_k, so that the k-th largest logit is the mask and all masked tokens are kept (with
# probability 0).  V below and above the fp32 list's 4096.
MASKS = [-1e9, -1e10, -1e30, "lowest"]


def masked(z, left, value):
    g = torch.Generator(device="cuda").manual_seed(z.shape[-1])
    keep = torch.randperm(z.shape[-1], generator=g, device="cuda")[:left]
    out = torch.full_like(z, torch.finfo(z.dtype).min if value == "lowest" else value)
    out[..., keep] = z[..., keep]
    return out, keep


@pytest.mark.parametrize("mask", MASKS)
@pytest.mark.parametrize("dtype", [BF, F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("V", [1000, 20003])
@pytest.mark.parametrize("shift", [0.0, -30.0], ids=["max_above_0", "max_below_0"])
def test_finite_masks(V, dtype, mask, shift):
    z, _ = masked((rows(V, dtype).float() + shift).to(dtype), 20, mask)
    for T in (0.3, 0.6, 1.0):
        for trunc in (dict(top_k=50), dict(top_k=50, top_p=0.95), dict(top_p=0.95)):
            check(z, trunc, T)


@pytest.mark.parametrize("V", [50, 20003])
@pytest.mark.parametrize("dtype", [BF, F32], ids=["bf16", "f32"])
@pytest.mark.parametrize("trunc", [dict(top_k=50), dict(top_k=25), dict(top_p=0.95), dict(top_k=25, top_p=0.95)], ids=["k50", "k25", "p95", "k25p95"])
def test_distributions_with_far_exponents(V, dtype, trunc):
    """z log2(e) / T beyond 2^20 (where fp32 loses the fraction), 2^24 (integers) and 1e9 (references): low temperatures, rows far from
    zero, rows of a mask only."""
    z = rows(V, dtype)
    for shift, temperatures in ((0.0, (1e-5, 1e-6, 1e-7, 1e-9)), (-40.0, (1e-6, 1e-9)), (3e6, (1.0, 0.1)), (-3e7, (1.0, 0.1))):
        for T in temperatures:
            check((z.float() + shift).to(dtype), trunc, T)
    for value in (-1e9, -1e30, torch.finfo(dtype).min, 1e30):
        check(torch.full_like(z, value), trunc, 0.6)


@pytest.mark.parametrize("V", [8192, 8193, 40000, 150001])
@pytest.mark.parametrize("top,spread,T", [(-2.0 ** -11, 0.002, 1e-3),        # the largest logits at the edge of the bins that share values
                                          (-0.25, 4.0, 1.0), (-9.0, 3.0, 0.6),
                                          (-478.0, 3.0, 1.0), (-490.0, 3.0, 1.0),      # bounds whose 32 values below end at the outermost bin
                                          (-505.0, 6.0, 1.0)])
@pytest.mark.parametrize("p", [0.9, 0.99])
def test_rows_of_negative_logits(V, top, spread, T, p):
    g = torch.Generator(device="cuda").manual_seed(V)
    z = (top - torch.rand((1, 4, V), generator=g, device="cuda") ** 2 * spread).to(BF)
    if V > 8192:
        z[0, 1, 8192:] = (z[0, 1, 8192:].float() * 0.5).to(BF)          # larger ones after the first slice
        z[0, 2, V - 1] = 0.0                                            # a logit of the other kind late in the row
        z[0, 3, V - 2] = 0.5
    check(z, dict(top_p=p), T)
