"""The training step, whose diversity term is taken from D^T D, against the same step in fp64: sizes around the staging of
the atoms, few atoms, many codes per row."""
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


def _step64(D, X, s, lr, beta):
    D, N = D.double(), D.shape[0]
    grad, loss = torch.zeros_like(D), 0.0
    for x in X.split(1 << 14):
        x = x.double()
        R, used = x, []
        for _ in range(s):
            corr = R @ D.T
            n = corr.abs().argmax(dim=1)
            c = corr.gather(1, n[:, None])
            R = R - c * D[n]
            used.append((n, c))
        loss += float((R * R).sum())
        for n, c in used:
            grad.index_add_(0, n, -2.0 * c * R)
    G = D @ D.T - torch.eye(N, dtype=torch.float64, device=D.device)
    W = D - lr * (grad + beta * 4.0 / N ** 2 * (G @ D))
    return torch.nn.functional.normalize(W, dim=1), loss, float((G * G).sum()) / N ** 2


@pytest.mark.parametrize("M,N,d,s", [(2000, 700, 128, 8), (1500, 5001, 64, 8), (131, 300, 128, 1), (140, 1, 64, 1), (210, 33, 128, 64), (0, 1, 128, 2),
                                     (0, 65, 64, 2), (0, 4100, 128, 2)])
def test_step_against_fp64(csr, M, N, d, s):
    g = torch.Generator(device=DEV).manual_seed(M + N)
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1).contiguous()
    if N > 60:                                              # popular atoms: many entries each
        D[:50] = torch.nn.functional.normalize(D[:50] + 2.0 * D[0], dim=1)
    X = torch.randn(M, d, device=DEV, generator=g)
    if M > 10 and N > 60:
        X[: M // 2] += 6.0 * D[0]
    lr, beta = 1e-5, 0.5
    want, l_mse, l_div = _step64(D, X, s, lr, beta)
    losses = torch.empty(2, dtype=torch.float64, device=DEV)
    before = D.clone()
    csr.csr_dict_train_step(D, X, s, lr, beta, mode=csr.CSR_MODE_FP32_EXACT, losses=losses)
    assert csr.csr_device_status() == csr.CSR_OK
    # fp32 errors x - x^ (128 eps of the row's norm at most, taken up by the sums), squared and summed in fp64; fp64 D^T D
    assert abs(float(losses[0]) - l_mse) <= 1e-5 * l_mse + 1e-12
    assert abs(float(losses[1]) - l_div) <= 1e-12 * (1.0 + l_div)
    # the step itself to 1e-4 of its largest displacement (fp32 sums of up to M s terms), the atoms to fp32
    moved = float((want - before.double()).abs().max())
    assert float((D.double() - want).abs().max()) <= 1e-4 * moved + 4 * 2.0 ** -24


def test_orthonormal_atoms_have_no_diversity_loss(csr):
    """N = d orthonormal atoms up to their fp32 rounding e: D D^T - I is of the order e, and so is what the step moves."""
    g = torch.Generator(device=DEV).manual_seed(1)
    D = torch.linalg.qr(torch.randn(128, 128, dtype=torch.float64, device=DEV, generator=g))[0].float().contiguous()
    want, _, l_div = _step64(D, torch.empty(0, 128, device=DEV), 1, 1.0, 1.0)
    losses = torch.empty(2, dtype=torch.float64, device=DEV)
    csr.csr_dict_train_step(D, torch.empty(0, 128, device=DEV), 1, 1.0, 1.0, losses=losses)
    assert 0.0 < l_div < 1e-14 and abs(float(losses[1]) - l_div) <= 1e-16
    assert float((D.double() - want).abs().max()) <= 2.0 ** -23
