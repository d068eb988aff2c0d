"""The exact mode's split engine (up to one row tile per SM, the dictionary split across the CTAs of a
row tile) and the plan that runs a last, partial wave of row tiles with it: the codes must be those
of the one-CTA-per-pair engine bit for bit, and the oracle's picks."""
import numpy as np
import pytest
import torch

from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def csr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2412_11741_b200 as m
    return m


def _np(t):
    return t.contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


# rows: one, around one tile, several slices per tile, one tile per SM and just over (two launches), a whole
# wave of pairs and a rest; atoms: one, two, around a 64-atom box, widths of 64 to 256 columns, several tiles
@pytest.mark.parametrize("M,N,d,s,dtype", [(1, 1, 128, 3, torch.float32), (2, 2, 64, 5, torch.bfloat16), (16, 8192, 128, 16, torch.bfloat16),
                                           (127, 63, 64, 4, torch.float16), (128, 65, 128, 4, torch.float32), (129, 129, 128, 6, torch.float16),
                                           (300, 1000, 64, 6, torch.bfloat16), (1500, 5001, 128, 8, torch.float32),
                                           (9473, 700, 128, 3, torch.bfloat16), (18944, 600, 64, 3, torch.bfloat16),
                                           (18945, 600, 128, 3, torch.float32), (24000, 513, 128, 2, torch.bfloat16),
                                           (38000, 300, 64, 2, torch.bfloat16), (57000, 300, 128, 2, torch.float16)])
def test_split_engine_equals_the_pair_engine(csr, M, N, d, s, dtype):
    g = torch.Generator(device=DEV).manual_seed(M + N)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1)
    X = torch.randn(M, d, device=DEV, generator=g)
    if N > 4:
        D[N // 2], D[N - 1] = D[1], -D[2]                 # equal correlations: the lower index wins
        X[0] = 3.0 * D[1]
    if N >= 129:                                          # more atoms inside the band than a sweep keeps track of
        D[20:60] = torch.nn.functional.normalize(D[20] + 1e-5 * torch.randn(40, d, device=DEV, generator=g), dim=1)
        X[M // 3] = 2.0 * D[30]
    if M > 2:
        X[M // 2] = 0.0
    D, X = D.contiguous(), X.to(dtype)
    idx, coef = csr.csr_encode_ex(D, X, s, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    assert csr.csr_device_status() == csr.CSR_OK
    csr.csr_set_option("exact_engine", 2)
    try:
        idx2, coef2 = csr.csr_encode_ex(D, X, s, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    finally:
        csr.csr_set_option("exact_engine", 0)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(idx), _np(idx2)) and torch.equal(coef, coef2)
    if M <= 1500:
        rep = parity.compare_exact(D.cpu().numpy(), X.float().cpu().numpy(), s, _np(idx), coef.cpu().numpy())
        assert rep.ok, rep.detail


@pytest.mark.parametrize("over,N,d", [(1, 1024, 128), (9, 1023, 64), (10, 1024, 128), (18, 2048, 64), (19, 2300, 128), (37, 4096, 64), (38, 4100, 128)])
def test_second_launch_of_single_tiles(csr, over, N, d):
    """More row tiles than SMs by `over`, on both sides of where the second launch has too few slices: the codes of pairs."""
    M = 128 * torch.cuda.get_device_properties(0).multi_processor_count + 128 * over - 5
    g = torch.Generator(device=DEV).manual_seed(M + N)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(M, d, device=DEV, generator=g).to(torch.bfloat16)
    idx, coef = csr.csr_encode_ex(D, X, 2, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    csr.csr_set_option("exact_engine", 2)
    try:
        idx2, coef2 = csr.csr_encode_ex(D, X, 2, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    finally:
        csr.csr_set_option("exact_engine", 0)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(idx), _np(idx2)) and torch.equal(coef, coef2)


def test_split_engine_writes_strided_codes_and_reads_strided_rows(csr):
    g = torch.Generator(device=DEV).manual_seed(3)
    D = torch.nn.functional.normalize(torch.randn(1000, 64, device=DEV, generator=g), dim=1).contiguous()
    wide = torch.randn(200, 128, device=DEV, generator=g)
    out_i = torch.full((200, 12), -1, dtype=torch.int16, device=DEV).view(torch.uint16)
    out_c = torch.full((200, 12), 7.0, device=DEV)
    csr.csr_encode_ex(D, wide[:, 64:], 6, mode=csr.CSR_MODE_FP32_EXACT, out_idx=out_i[:, 3:9], out_coef=out_c[:, 3:9])
    idx, coef = csr.csr_encode_ex(D, wide[:, 64:].contiguous(), 6, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(out_i)[:, 3:9], _np(idx)) and torch.equal(out_c[:, 3:9], coef)
    assert np.all(_np(out_i)[:, :3] == 0xFFFF) and np.all(_np(out_i)[:, 9:] == 0xFFFF) and bool((out_c[:, 9:] == 7.0).all())


def test_split_engine_bounded_wait_runs_out_and_recovers(csr):
    """The CTAs of a row tile wait for one another in global memory: with no time to wait the call
    returns, the status word reports it, and the next call is whole again."""
    g = torch.Generator(device=DEV).manual_seed(4)
    D = torch.nn.functional.normalize(torch.randn(2000, 128, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(500, 128, device=DEV, generator=g)
    want = csr.csr_encode_ex(D, X, 4, mode=csr.CSR_MODE_FP32_EXACT)
    assert csr.csr_device_status() == csr.CSR_OK
    csr.csr_set_option("wait_limit_ns", 0)
    try:
        csr.csr_encode_ex(D, X, 4, mode=csr.CSR_MODE_FP32_EXACT)
        assert csr.csr_device_status() == csr.CSR_ERR_TIMEOUT
    finally:
        csr.csr_set_option("wait_limit_ns", 2_000_000_000)
    got = csr.csr_encode_ex(D, X, 4, mode=csr.CSR_MODE_FP32_EXACT)
    assert csr.csr_device_status() == csr.CSR_OK
    assert np.array_equal(_np(got[0]), _np(want[0])) and torch.equal(got[1], want[1])


def test_split_engine_captured_in_a_cuda_graph(csr):
    g = torch.Generator(device=DEV).manual_seed(5)
    D = torch.nn.functional.normalize(torch.randn(3000, 128, device=DEV, generator=g), dim=1).contiguous()
    X1, X2 = (torch.randn(100, 128, device=DEV, generator=g) for _ in range(2))
    want = [csr.csr_encode_ex(D, x, 5, mode=csr.CSR_MODE_FP32_EXACT) for x in (X1, X2)]
    X = X1.clone()
    idx = torch.zeros((100, 5), dtype=torch.int16, device=DEV).view(torch.uint16)
    coef = torch.zeros((100, 5), dtype=torch.float16, device=DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        csr.csr_encode_ex(D, X, 5, mode=csr.CSR_MODE_FP32_EXACT, out_idx=idx, out_coef=coef)
    for x, w in ((X1, want[0]), (X2, want[1])):
        X.copy_(x)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(_np(idx), _np(w[0])) and torch.equal(coef, w[1])
    assert csr.csr_device_status() == csr.CSR_OK
    del graph
