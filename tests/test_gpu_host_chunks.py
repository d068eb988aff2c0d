"""The host entry points cut their rows into two halves of a wave of row-tile pairs and whole waves: the codes and rows of every size
around the cuts are those of one device call."""
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


@pytest.mark.parametrize("waves,extra", [(0.5, 0), (0.5, 1), (1, 0), (1, 1), (2, -1), (2, 1), (9, 130)])
@pytest.mark.parametrize("prepared", [False, True])
def test_chunks_give_the_codes_of_one_call(csr, waves, extra, prepared):
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 256
    M, N, d, s = int(waves * wave) + extra, 300, 64, 3
    g = torch.Generator(device=DEV).manual_seed(M)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(M, d, device=DEV, generator=g).to(torch.bfloat16)
    h = csr.csr_dict_create(D) if prepared else None
    want_i, want_c = csr.csr_encode_ex(D, X, s, dict=h)
    want_x = csr.csr_reconstruct_ex(D, want_i, want_c, dict=h, out_dtype=torch.bfloat16)
    torch.cuda.synchronize()
    idx = torch.empty(M, s, dtype=torch.uint16, pin_memory=True)
    coef = torch.empty(M, s, dtype=torch.float16, pin_memory=True)
    back = torch.empty(M, d, dtype=torch.bfloat16, pin_memory=True)
    csr.csr_encode_host(D, X.cpu().pin_memory(), s, idx, coef, dict=h)
    csr.csr_reconstruct_host(D, idx, coef, back, dict=h)
    assert csr.csr_device_status() == csr.CSR_OK
    assert torch.equal(idx.view(torch.int16), want_i.view(torch.int16).cpu()) and torch.equal(coef, want_c.cpu())
    assert torch.equal(back, want_x.cpu())
    if h:
        csr.csr_dict_destroy(h)
