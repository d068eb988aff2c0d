"""The de-sparse kernel's ways of taking a row (four, three or any number of entries at a time) and its
units of 16, 8 or 4 rows, around the sizes where they change, against a plain sum in the stored
order (fp32, the same order of additions: the bound is one rounding per addition)."""
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


@pytest.mark.parametrize("M,N,d,s,out,cd,handle", [
    (1, 1, 64, 1, torch.float32, torch.float32, False), (3, 5, 128, 3, torch.float32, torch.float16, True),
    (17, 100, 128, 6, torch.float32, torch.float32, False), (77777, 501, 128, 6, torch.float32, torch.float16, False),
    (60001, 501, 64, 9, torch.float32, torch.float16, True), (60001, 501, 64, 6, torch.float32, torch.float32, True),
    (75777, 300, 128, 4, torch.float32, torch.float16, False), (75776, 300, 128, 5, torch.float32, torch.float16, False),
    (57000, 300, 128, 8, torch.float32, torch.float16, True), (30001, 300, 64, 12, torch.float32, torch.float32, False)])
def test_every_path_and_unit(csr, M, N, d, s, out, cd, handle):
    g = torch.Generator(device=DEV).manual_seed(M + s)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    i = torch.randint(0, N, (M, s), device=DEV, generator=g)
    idx = i.to(torch.int16).view(torch.uint16)
    coef = torch.randn(M, s, device=DEV, generator=g).to(cd)
    h = csr.csr_dict_create(D) if handle else None
    X = torch.full((M + 1, d), 7.0, dtype=out, device=DEV)
    csr.csr_reconstruct_ex(D, idx, coef, X_hat=X[:M], dict=h)
    # codes inside wider arrays take the element-wise staging: the same values
    wide_i = torch.zeros((M, s + 3), dtype=torch.int16, device=DEV).view(torch.uint16)
    wide_c = torch.zeros((M, s + 3), dtype=cd, device=DEV)
    wide_i.view(torch.int16)[:, 1:s + 1], wide_c[:, 1:s + 1] = idx.view(torch.int16), coef
    X2 = csr.csr_reconstruct_ex(D, wide_i[:, 1:s + 1], wide_c[:, 1:s + 1], out_dtype=out, dict=h)
    if h is not None:
        csr.csr_dict_destroy(h)
    assert bool((X[M] == 7.0).all()) and torch.equal(X[:M], X2)
    A = (D.half() if handle else D).double()
    ref = torch.zeros(M, d, dtype=torch.float64, device=DEV)
    mag = torch.zeros_like(ref)
    for q in range(s):
        term = coef[:, q:q + 1].double() * A[i[:, q]]
        ref += term
        mag += term.abs()
    assert bool(((X[:M].double() - ref).abs() <= s * 2.0 ** -24 * mag + 1e-30).all())
