"""Fast encodes that convert their dictionary first: the encoder's CTAs come up beside the conversion and wait for it.  Each kind of
launch (a handful of rows, clusters, single row tiles, pairs) must see the dictionary of its own call, also in a captured graph."""
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


def _unit(g, n, d):
    return torch.nn.functional.normalize(torch.randn(n, d, device=DEV, generator=g), dim=1).contiguous()


# (atoms not a multiple of eight: the conversion writes the padding too)
@pytest.mark.parametrize("M,N,d", [(8, 8191, 128), (500, 4099, 64), (4160, 1027, 128), (18944, 301, 64), (40000, 513, 128)])
def test_every_call_sees_its_own_dictionary(csr, M, N, d):
    g = torch.Generator(device=DEV).manual_seed(M)
    X = torch.randn(M, d, device=DEV, generator=g)
    dicts = [_unit(g, N, d) for _ in range(4)]
    want = []
    for D in dicts:                                         # prepared dictionaries: no conversion in front of the encoder
        h = csr.csr_dict_create(D)
        torch.cuda.synchronize()
        want.append(csr.csr_encode_ex(D, X, 4, dict=h))
        torch.cuda.synchronize()
        csr.csr_dict_destroy(h)
    got = [csr.csr_encode_ex(D, X, 4) for D in dicts]       # one after the other in the same scratch, nothing waited for
    torch.cuda.synchronize()
    assert csr.csr_device_status() == csr.CSR_OK
    for (i0, c0), (i1, c1) in zip(want, got):
        assert torch.equal(i0.view(torch.int16), i1.view(torch.int16)) and torch.equal(c0, c1)
    D, idx, coef = dicts[0].clone(), torch.empty_like(got[0][0]), torch.empty_like(got[0][1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        csr.csr_encode_ex(D, X, 4, out_idx=idx, out_coef=coef)
    for k in (2, 1):
        D.copy_(dicts[k])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(idx.view(torch.int16), want[k][0].view(torch.int16)) and torch.equal(coef, want[k][1])
    assert csr.csr_device_status() == csr.CSR_OK
    del graph
