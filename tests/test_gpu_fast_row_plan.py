"""The fast encoder's plan of a call's rows (whole waves of pairs of row tiles, then single row tiles with
one or more CTAs each): the codes are those of pairs only, bit for bit, around the sizes where the
plan changes (one row, one tile, one tile per SM, a wave of pairs, what is left over)."""
import numpy as np
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


def _np(t):
    return t.contiguous().view(torch.int16).cpu().numpy()


@pytest.mark.parametrize("d,N", [(128, 200), (128, 1024), (128, 2500), (64, 600), (64, 9000)])
@pytest.mark.parametrize("M", [1, 8, 9, 40, 127, 129, 500, 1025, 4160, 9473, 18944, 18945, 26000, 37888, 38000, 60000])
def test_plan_gives_the_codes_of_pairs(csr, d, N, M):
    g = torch.Generator(device=DEV).manual_seed(M + N)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(M, d, device=DEV, generator=g).to(torch.bfloat16)
    if N > 600:
        D[N - 1], X[0] = D[5], 3.0 * D[5].to(torch.bfloat16)
    X[M // 2] = 0.0
    out_i = torch.full((M + 1, 3), -1, dtype=torch.int16, device=DEV).view(torch.uint16)
    out_c = torch.full((M + 1, 3), 7.0, device=DEV)
    csr.csr_encode_ex(D, X, 3, out_idx=out_i[:M], out_coef=out_c[:M])
    assert csr.csr_device_status() == csr.CSR_OK
    csr.csr_set_option("fast_split", 1)
    try:
        idx, coef = csr.csr_encode_ex(D, X, 3, coef_dtype=torch.float32)
    finally:
        csr.csr_set_option("fast_split", 0)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(out_i)[:M], _np(idx)) and torch.equal(out_c[:M], coef)
    assert np.all(_np(out_i)[M] == -1) and bool((out_c[M] == 7.0).all())


def test_single_tiles_bounded_wait_runs_out_and_recovers(csr):
    g = torch.Generator(device=DEV).manual_seed(4)
    D = torch.nn.functional.normalize(torch.randn(4096, 128, device=DEV, generator=g), dim=1).contiguous()
    for M in (100, 3000, 15000):
        X = torch.randn(M, 128, device=DEV, generator=g).to(torch.bfloat16)
        want = csr.csr_encode_ex(D, X, 4)
        assert csr.csr_device_status() == csr.CSR_OK
        csr.csr_set_option("wait_limit_ns", 0)
        try:
            csr.csr_encode_ex(D, X, 4)
            assert csr.csr_device_status() == csr.CSR_ERR_TIMEOUT
        finally:
            csr.csr_set_option("wait_limit_ns", 2_000_000_000)
        got = csr.csr_encode_ex(D, X, 4)
        assert csr.csr_device_status() == csr.CSR_OK
        assert np.array_equal(_np(got[0]), _np(want[0])) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("M,N,d,s", [(8, 8192, 128, 6), (120, 3000, 64, 5), (40, 1000, 128, 4), (1500, 4096, 128, 4), (3000, 2048, 64, 4)])
def test_clusters_that_give_up_leave_no_words_behind(csr, M, N, d, s):
    """The CTAs of a cluster write into one another's shared memory.  Calls that give up at once, each followed
    at once on the same SMs by a whole call: that one's codes are right every time."""
    g = torch.Generator(device=DEV).manual_seed(M)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(M, d, device=DEV, generator=g).to(torch.bfloat16)
    want_i, want_c = csr.csr_encode_ex(D, X, s)
    assert csr.csr_device_status() == csr.CSR_OK
    gave_up = torch.zeros(1, dtype=torch.int32, device=DEV)
    whole = []
    try:
        for _ in range(8):
            csr.csr_set_option("wait_limit_ns", 0)
            csr.csr_encode_ex(D, X, s, dev_status=gave_up)
            csr.csr_set_option("wait_limit_ns", 2_000_000_000)
            whole.append(csr.csr_encode_ex(D, X, s))
    finally:
        csr.csr_set_option("wait_limit_ns", 2_000_000_000)
    assert csr.csr_device_status() == csr.CSR_OK          # of the whole calls: the others have a word of their own
    assert int(gave_up.item()) != 0
    for idx, coef in whole:
        assert np.array_equal(_np(idx), _np(want_i)) and torch.equal(coef, want_c)


@pytest.mark.parametrize("d,N", [(64, 1000), (64, 2304), (64, 5000), (128, 1000)])
@pytest.mark.parametrize("M", [8, 50, 200])
def test_rows_that_are_not_finite_get_the_codes_of_pairs_too(csr, d, N, M):
    """An infinite channel makes an atom's correlation infinite, or NaN where the atom does not use the channel: groups of
    atoms with some NaNs and with nothing but NaNs."""
    g = torch.Generator(device=DEV).manual_seed(M + N)
    D = torch.randn(N, d, device=DEV, generator=g)
    D[::3, 5] = 0.0
    D[40:64, 5] = 0.0
    D = torch.nn.functional.normalize(D, dim=1).contiguous()
    X = torch.randn(M, d, device=DEV, generator=g)
    X[1, 5], X[3, 5], X[4] = float("inf"), -float("inf"), float("nan")
    X[6, 4], X[6, 5] = float("inf"), -float("inf")
    X = X.to(torch.bfloat16)
    idx, coef = csr.csr_encode_ex(D, X, 4, coef_dtype=torch.float32)
    csr.csr_set_option("fast_split", 1)
    try:
        idx2, coef2 = csr.csr_encode_ex(D, X, 4, coef_dtype=torch.float32)
    finally:
        csr.csr_set_option("fast_split", 0)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(idx), _np(idx2))
    assert bool(((coef == coef2) | (coef.isnan() & coef2.isnan())).all())


@pytest.mark.parametrize("d,N,rows", [(128, 4096, (128, 128)), (128, 1024, (512, 40, 9472, 1025)), (64, 2500, (9000, 9000, 9000, 9000)),
                                      (128, 2000, (30000, 8, 700)), (64, 1000, (1024,) * 6), (128, 300, (40000, 38000))])
def test_grouped_problems_get_the_codes_of_pairs(csr, d, N, rows):
    """Problems side by side plan for their share of the GPU: other splits than alone, the same codes."""
    g = torch.Generator(device=DEV).manual_seed(sum(rows))
    problems, want = [], []
    for M in rows:
        D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
        X = torch.randn(M, d, device=DEV, generator=g).to(torch.bfloat16)
        problems.append((D, X, 3, torch.full((M, 3), -1, dtype=torch.int16, device=DEV).view(torch.uint16),
                         torch.full((M, 3), 7.0, dtype=torch.float16, device=DEV), csr.csr_dict_create(D)))
    csr.csr_set_option("fast_split", 1)
    try:
        want = [csr.csr_encode_ex(D, X, s) for D, X, s, _, _, _ in problems]
    finally:
        csr.csr_set_option("fast_split", 0)
    csr.csr_encode_grouped(problems)
    assert csr.csr_device_status() == csr.CSR_OK
    for (_, _, _, idx, coef, h), (i, c) in zip(problems, want):
        assert np.array_equal(_np(idx), _np(i)) and torch.equal(coef, c)
        csr.csr_dict_destroy(h)
