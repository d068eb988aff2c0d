"""The exact mode's tensor-core engines on rows of any norm: a row times a power of two has the row's codes
and its coefficients times that power, to the bit, because fp64 arithmetic scales exactly."""
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


@pytest.fixture(params=["split", "pairs"])
def engine(request, csr):
    csr.csr_set_option("exact_engine", 2 if request.param == "pairs" else 0)
    yield request.param
    csr.csr_set_option("exact_engine", 0)


def _unit(x):
    return torch.nn.functional.normalize(x, dim=1)


def _encode(csr, D, X, s):
    idx, coef = csr.csr_encode_ex(D, X, s, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
    assert csr.csr_device_status() == csr.CSR_OK
    return idx.view(torch.int16), coef


@pytest.mark.parametrize("M,N,d,s,dtype", [(100, 2000, 128, 6, torch.float32), (200, 513, 64, 4, torch.bfloat16), (3000, 700, 128, 5, torch.float32)])
def test_codes_do_not_depend_on_the_scale_of_a_row(csr, engine, M, N, d, s, dtype):
    g = torch.Generator(device=DEV).manual_seed(M)
    D = _unit(torch.randn(N, d, device=DEV, generator=g))
    D[20:60] = _unit(D[20] + 1e-5 * torch.randn(40, d, device=DEV, generator=g))       # more candidates than a sweep keeps track of
    X = torch.randn(M, d, device=DEV, generator=g).to(dtype)
    X[M // 3] = (2.0 * D[30] + 0.05 * torch.randn(d, device=DEV, generator=g)).to(dtype)
    # every element and coefficient stays a normal fp32 number
    powers = torch.tensor([-100, -90, -83, -60, -20, 0, 20, 60, 83, 100, 119], device=DEV)
    scale = torch.ldexp(torch.ones(M, device=DEV), powers[torch.arange(M, device=DEV) % len(powers)])
    scaled = (X.float() * scale[:, None]).to(dtype)
    assert bool((scaled.float() / scale[:, None] == X.float()).all())
    want_i, want_c = _encode(csr, D.contiguous(), X, s)
    got_i, got_c = _encode(csr, D.contiguous(), scaled, s)
    assert float(want_c.abs().min()) > 2.0 ** -20
    assert torch.equal(got_i, want_i)
    assert torch.equal(got_c, want_c * scale[:, None])


def test_residual_that_collapses_in_one_step(csr, engine):
    """x = e_0 + 2^-100 y, with e_0 an atom and no other atom or y using channel 0: the first pick leaves 2^-100 y, thirty
    orders of magnitude smaller, and the picks after it are those of y."""
    g = torch.Generator(device=DEV).manual_seed(1)
    M, N, d, s = 150, 1500, 128, 5
    D = torch.randn(N, d, device=DEV, generator=g)
    D[:, 0] = 0.0
    D[0] = 0.0
    D = _unit(D)
    D[0, 0] = 1.0
    Y = torch.randn(M, d, device=DEV, generator=g)
    Y[:, 0] = 0.0
    X = Y * 2.0 ** -100
    X[:, 0] = 1.0
    want_i, want_c = _encode(csr, D.contiguous(), Y.contiguous(), s)
    got_i, got_c = _encode(csr, D.contiguous(), X.contiguous(), s + 1)
    assert bool((got_i[:, 0] == 0).all()) and bool((got_c[:, 0] == 1.0).all())
    assert torch.equal(got_i[:, 1:], want_i) and torch.equal(got_c[:, 1:], want_c * 2.0 ** -100)


@pytest.mark.parametrize("M", [64, 700, 3000])
def test_rows_that_are_not_finite_leave_the_others_alone(csr, engine, M):
    g = torch.Generator(device=DEV).manual_seed(M)
    D = _unit(torch.randn(1000, 128, device=DEV, generator=g)).contiguous()
    X = torch.randn(M, 128, device=DEV, generator=g)
    bad = X.clone()
    bad[5, 3], bad[9], bad[17, 100] = float("nan"), float("inf"), -float("inf")
    good = torch.ones(M, dtype=torch.bool, device=DEV)
    good[[5, 9, 17]] = False
    (i0, c0), (i1, c1) = _encode(csr, D, X, 6), _encode(csr, D, bad, 6)
    assert torch.equal(i0[good], i1[good]) and torch.equal(c0[good], c1[good])
    assert bool(((i1.long() & 0xFFFF) < 1000).all())
