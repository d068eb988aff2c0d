"""Attention from the codes over the shapes at which its launch plan changes (heads per group, streams
and chunks against SMs, codes fetched ahead or not, row tiles, slices) against fp64 sums of the
restored rows."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def csr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2412_11741_b200 as m
    return m


def _inputs(B, H, T, Nk, Nv, d, sk, sv, qd, cd):
    g = torch.Generator(device=DEV).manual_seed(B * 1000 + T)
    unit = lambda n: torch.nn.functional.normalize(torch.randn(n, d, device=DEV, generator=g), dim=1).contiguous()
    codes = lambda n, s: (torch.randint(0, n, (B, T, s), device=DEV, generator=g).to(torch.int16).view(torch.uint16),
                          torch.randn(B, T, s, device=DEV, generator=g).to(cd))
    return unit(Nk), unit(Nv), torch.randn(B, H, d, device=DEV, generator=g).to(qd), codes(Nk, sk), codes(Nv, sv)


def _rows(D, idx, coef):
    return (coef.double()[:, :, None] * D.double()[idx.view(torch.int16).long() & 0xFFFF]).sum(1)


@pytest.mark.parametrize("B,H,T,Nk,Nv,d,sk,sv,qd,cd", [
    (1, 1, 1, 1, 1, 64, 1, 1, torch.float32, torch.float16),
    (8, 4, 4099, 8192, 8192, 128, 16, 16, torch.bfloat16, torch.float16),      # one head per group: more items than SMs
    (3, 5, 1025, 1001, 777, 64, 8, 6, torch.float16, torch.float32),           # odd sizes, fp32 coefficients
    (40, 4, 2050, 4097, 3000, 128, 8, 16, torch.float32, torch.float16),       # whole groups, more than 32 rows, two slices and more
    (70, 6, 1100, 600, 901, 64, 16, 8, torch.bfloat16, torch.float16),         # six heads in groups of eight
    (150, 3, 513, 2000, 1500, 128, 3, 24, torch.float16, torch.float16),       # a padded head; codes not fetched ahead
    (2, 1, 20000, 49152, 300, 128, 8, 8, torch.float32, torch.float16),        # the largest table one head may have
])
def test_decode_attention_over_the_plans(csr, B, H, T, Nk, Nv, d, sk, sv, qd, cd):
    Dk, Dv, Q, (ki, kc), (vi, vc) = _inputs(B, H, T, Nk, Nv, d, sk, sv, qd, cd)
    scale = 1.0 / math.sqrt(d)
    out, w = csr.csr_decode_attention(Dk, Dv, Q, ki, kc, vi, vc, scale)
    scores = csr.csr_key_scores(Dk, Q, ki, kc, scale)
    mix = csr.csr_value_mix(Dv, w, vi, vc)
    again = csr.csr_decode_attention(Dk, Dv, Q, ki, kc, vi, vc, scale)
    assert torch.equal(out, again[0]) and torch.equal(w, again[1])             # the same bits on every run
    for b in range(0, B, max(1, B // 4)):
        ref_s = Q[b].double() @ _rows(Dk, ki[b], kc[b]).T * scale
        W = torch.softmax(ref_s, -1)
        ref = W @ _rows(Dv, vi[b], vc[b])
        # a score's fp32 sums: 2e-6 of sum |coef| ||q|| scale (atoms have norm 1); a weight's relative error is at most
        # twice the largest score error plus the exponential's own few ulp
        ds = 2e-6 * kc[b].double().abs().sum(-1)[None, :] * Q[b].double().norm(dim=1)[:, None] * scale
        assert bool(((scores[b] - ref_s).abs() <= ds).all())
        dw = 2 * ds.max(dim=1, keepdim=True).values + 2e-6
        assert bool(((w[b] - W).abs() <= W * dw).all())
        # an output: the weights' error, fp32 rounding, and half a grid step per term (2^-29 of S U, S <= 1)
        l1 = vc[b].double().abs().sum(-1)
        tol = (W * l1).sum(-1, keepdim=True) * (dw + 4e-6) + T * sv * 2.0 ** -30 * l1.max()
        assert bool(((out[b] - ref).abs() <= tol).all()) and bool(((mix[b] - ref).abs() <= tol).all())


def test_infinities_and_nans_stay_in_their_rows(csr):
    B, H, T, N, d, s = 5, 4, 900, 700, 64, 8
    Dk, Dv, Q, (ki, kc), (vi, vc) = _inputs(B, H, T, N, N, d, s, s, torch.float32, torch.float16)
    clean = csr.csr_decode_attention(Dk, Dv, Q, ki, kc, vi, vc, 0.125)
    clean = [t.clone() for t in clean]
    Q2, vc2 = Q.clone(), vc.clone()
    Q2[1, 2, 3] = float("nan")                            # one row of weights
    vc2[3, 17, 1] = float("inf")                          # one stream of outputs
    out, w = csr.csr_decode_attention(Dk, Dv, Q2, ki, kc, vi, vc2, 0.125)
    assert bool(w[1, 2].isnan().all()) and bool(out[1, 2].isnan().all())
    assert not bool(torch.isfinite(out[3]).all())
    for b in (0, 2, 4):
        assert torch.equal(out[b], clean[0][b]) and torch.equal(w[b], clean[1][b])
    assert torch.equal(w[3], clean[1][3])
    for h in (0, 1, 3):
        assert torch.equal(w[1, h], clean[1][1, h]) and bool(torch.isfinite(out[1, h]).all())


def test_overlapped_launches_in_a_cuda_graph(csr):
    """The kernels of a decoding step overlap (each waits for the one before it on the device): captured and
    replayed on new queries, and after another call has used the same scratch, the step returns
    what it returns alone."""
    Dk, Dv, Q, (ki, kc), (vi, vc) = _inputs(6, 4, 3000, 2000, 1500, 128, 16, 8, torch.float32, torch.float16)
    Q2 = Q.flip(0).contiguous()
    want = [tuple(t.clone() for t in csr.csr_decode_attention(Dk, Dv, q, ki, kc, vi, vc, 0.09)) for q in (Q, Q2)]
    q, w, out = Q.clone(), torch.empty(6, 4, 3000, device=DEV), torch.empty(6, 4, 128, device=DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        csr.csr_decode_attention(Dk, Dv, q, ki, kc, vi, vc, 0.09, weights=w, out=out)
    for _ in range(3):
        for src, (o, ww) in ((Q, want[0]), (Q2, want[1])):
            q.copy_(src)
            graph.replay()
            csr.csr_key_scores(Dk, Q2, ki, kc, 0.5)
            torch.cuda.synchronize()
            assert torch.equal(out, o) and torch.equal(w, ww)
    del graph


@pytest.mark.parametrize("T,at", [(2, 0), (900, 0), (900, 512), (900, 700), (4099, 3071)])
@pytest.mark.parametrize("B,H,s", [(3, 4, 8), (40, 2, 6)])
def test_one_nan_or_infinite_score_is_softmaxed_like_any_other(csr, B, H, s, T, at):
    """One token's key coefficient is NaN, another stream's is infinite (scores of +Inf and -Inf, by the sign of q . d):
    the weights are NaN where the softmax of the scores is, wherever in the row the token stands."""
    Dk, Dv, Q, (ki, kc), (vi, vc) = _inputs(B, H, T, 300, 200, 64, s, s, torch.float32, torch.float16)
    kc[0, at, 1], kc[2, at, 3] = float("nan"), float("inf")
    out, w = csr.csr_decode_attention(Dk, Dv, Q, ki, kc, vi, vc, 0.125)
    scores = csr.csr_key_scores(Dk, Q, ki, kc, 0.125)
    assert bool(scores[0, :, at].isnan().all()) and bool(scores[2, :, at].isinf().all()) and not bool(scores[1].isnan().any())
    want = torch.softmax(scores.double(), -1)
    assert bool(w[0].isnan().all()) and bool(out[0].isnan().all())
    assert torch.equal(w.isnan(), want.isnan())
    # the exponentials' few ulp, and their arguments' rounding
    torch.testing.assert_close(w.double(), want, rtol=2e-5, atol=1e-30, equal_nan=True)


@pytest.mark.parametrize("B,H,T,N,d,s,unit", [(10, 64, 16384, 500, 64, 8, 2048), (18, 64, 6000, 9000, 128, 16, 1024), (4, 32, 9000, 24000, 64, 8, 1024)])
def test_value_grid_does_not_coarsen_with_the_number_of_head_groups(csr, B, H, T, N, d, s, unit):
    """`unit`: the tokens of a piece when all SMs share the streams' tokens and a piece takes all heads.  A grid of 29 bits
    over such a piece's bound has steps of at most 2^-28 S U (the scale is a power of two); T s terms, each half a
    step off at most, give an output this error in the root mean square."""
    _, Dv, _, _, (vi, vc) = _inputs(B, H, T, 2, N, d, 1, s, torch.float32, torch.float16)
    g = torch.Generator(device=DEV).manual_seed(N)
    W = torch.rand(B, H, T, device=DEV, generator=g)
    W /= W.sum(-1, keepdim=True)
    out = csr.csr_value_mix(Dv, W, vi, vc)
    for b in (0, B - 1):
        ref = W[b].double() @ _rows(Dv, vi[b], vc[b])
        U = float(vc[b].double().abs().sum(-1).max())
        S = float(torch.stack([w.sum(-1).max() for w in W[b].double().split(unit, dim=-1)]).max())
        bound = 2.0 ** -28 * S * U * math.sqrt(T * s / (12.0 * d))
        rms = float((out[b] - ref).pow(2).mean().sqrt())
        assert rms <= bound + 1e-6 * float(ref.pow(2).mean().sqrt()), (rms, bound)


@pytest.mark.parametrize("B,H,T,N,s", [(64, 4, 16384, 8192, 16), (8, 4, 4099, 8192, 16), (3, 64, 8000, 4096, 8)])
def test_weights_of_a_row_add_up_to_one_on_average(csr, B, H, T, N, s):
    """A row's weights share the error of its sum of exponentials, which is put together from parts with maxima of their
    own.  Roundings go either way: over the rows, the weights' sums miss 1 by less than half an fp32 ulp."""
    Dk, Dv, Q, (ki, kc), (vi, vc) = _inputs(B, H, T, N, N, 128, s, s, torch.float32, torch.float16)
    _, w = csr.csr_decode_attention(Dk, Dv, Q, ki, kc, vi, vc, 2.0 / math.sqrt(128))
    assert abs(float((w.double().sum(-1) - 1.0).mean())) < 2.0 ** -24
