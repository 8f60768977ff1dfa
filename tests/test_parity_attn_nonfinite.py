"""GPU parity: scores that are not finite numbers.  A NaN or +inf score makes the rows that see it NaN, as softmax in floating point
does, wherever in a 64-key step its key lies and however many steps the row has; a -inf score takes no part, and a row with no
other is zero.  Rows and heads that do not see such a key keep their values."""
import pytest
import torch

from paper_2604_16498_b200 import binding

pytestmark = pytest.mark.gpu

SIZES = [(40, torch.bfloat16), (64, torch.bfloat16), (64, torch.float16), (80, torch.bfloat16), (128, torch.bfloat16), (128, torch.float16),
         (192, torch.bfloat16)]


def _run(q, k, v, mask=0):
    out = (binding.attn_fused_f16 if q.dtype == torch.float16 else binding.attn_fused)(q, k, v, mask)
    binding.check_status()
    return out.float()


def _inputs(B, H, Sq, Skv, D, dtype):
    g = torch.Generator(device="cuda").manual_seed(91)
    mk = lambda s: torch.randn((B, H, s, D), generator=g, device="cuda").to(dtype)
    return mk(Sq), mk(Skv), mk(Skv)


def _each_key(D, dtype, Skv, value, H=2):
    """Batch entry b has `value` in key b of head 0; the others are left alone.  Two rows of queries, positive ones."""
    q, k, v = _inputs(Skv, H, 2, Skv, D, dtype)
    q = q.abs() + 0.125
    clean = _run(q, k, v)
    for b in range(Skv):
        k[b, 0, b] = value
    return q, k, v, clean, _run(q, k, v)


@pytest.mark.parametrize("D,dtype", SIZES)
@pytest.mark.parametrize("Skv", [64, 192])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_nan_or_inf_score_makes_the_row_nan_at_every_key(D, dtype, Skv, value):
    *_, clean, got = _each_key(D, dtype, Skv, value)
    lost = [b for b in range(Skv) if not got[b, 0].isnan().all()]
    assert not lost, f"keys whose score was dropped: {lost}"
    assert torch.equal(got[:, 1], clean[:, 1])


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_the_same_in_many_short_tiles(value):
    """More tiles than run at once: 192 x 8."""
    *_, clean, got = _each_key(64, torch.bfloat16, 192, value, 8)
    lost = [b for b in range(192) if not got[b, 0].isnan().all()]
    assert not lost, f"keys whose score was dropped: {lost}"
    assert torch.equal(got[:, 1:], clean[:, 1:])


@pytest.mark.parametrize("D,dtype", SIZES)
def test_a_nan_reaches_the_rows_that_see_it_and_no_others(D, dtype):
    q, k, v = _inputs(1, 2, 200, 200, D, dtype)
    clean = _run(q, k, v, binding.MASK_CAUSAL)
    for j in (5, 37, 70, 131):
        kk = k.clone()
        kk[0, 0, j, D - 1] = float("nan")
        got = _run(q, kk, v, binding.MASK_CAUSAL)
        assert got[0, 0, j:].isnan().all() and torch.equal(got[0, 1], clean[0, 1])
        assert (got[0, 0, :j] - clean[0, 0, :j]).abs().max() <= 2e-2  # the same values, a step's exponentials by the other unit


@pytest.mark.parametrize("D,dtype", SIZES)
@pytest.mark.parametrize("Skv", [64, 192])
def test_scores_of_minus_infinity_take_no_part(D, dtype, Skv):
    q, k, v = _inputs(Skv, 2, 2, Skv, D, dtype)
    q = q.abs() + 0.125
    clean = _run(q, k, v)
    k[:, 0] = float("-inf")
    none = _run(q, k, v)
    assert (none[:, 0] == 0).all() and torch.equal(none[:, 1], clean[:, 1])
    for b in range(Skv):  # one finite score, at key b
        k[b, 0, b] = 0.0
    one = _run(q, k, v)
    i = torch.arange(Skv, device="cuda")
    want = v[i, 0, i].float()[:, None, :].expand(-1, 2, -1)
    # beside it, each other key weighs at most 2^-125
    assert torch.equal(one[:, 0], want) and torch.equal(one[:, 1], clean[:, 1])
