"""The training step's gradient at numbers of entries per row that the smaller tests leave out: a last trip of the
loop over a row's codes that is not whole, more codes than a warp has lanes, the most there may be."""
import numpy as np
import pytest
import torch

from oracle import csr_oracle as orc
from paper_2412_11741_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("N,d,M,s", [(200, 128, 300, 11), (300, 64, 200, 31), (150, 128, 130, 33), (120, 64, 150, 45), (256, 128, 100, 64), (90, 64, 70, 64)])
def test_training_step_with_many_codes_per_row(N, d, M, s):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2412_11741_b200 as csr
    rng = np.random.default_rng(N + s)
    D0 = wl.normalise_rows(rng.standard_normal((N, d)).astype(np.float32))
    X = rng.standard_normal((M, d)).astype(np.float32)
    lr, beta = 1e-3, 0.7
    want_D, l_mse, l_div, res = orc.dict_train_step(D0, X, s, lr, beta)
    assert res.gap.min() > 1e-9                              # no tie in this batch: same codes on both sides
    Dd = torch.from_numpy(D0.copy()).to(DEV)
    losses = csr.csr_dict_train_step(Dd, torch.from_numpy(X).to(DEV), s, lr, beta).cpu().numpy()
    assert csr.csr_device_status() == csr.CSR_OK
    # An error of the gradient, channel by channel: e = x - sum c d takes s fp32 additions of values below A = |x| + sum |c d|,
    # an atom's n terms 2 c e are added in any order; the step adds lr times that, ReNorm and the diversity term a few ulp.
    idx, coef = res.idx.astype(np.int64), np.abs(res.coef)
    A = np.abs(X) + np.einsum("ms,msd->md", coef, np.abs(D0[idx]))
    S, T, n = np.zeros((N, d)), np.zeros((N, d)), np.zeros(N)
    e = np.abs(X.astype(np.float64) - np.einsum("ms,msd->md", res.coef, D0[idx].astype(np.float64)))
    for g in range(s):
        np.add.at(S, idx[:, g], 2 * coef[:, g, None] * A)
        np.add.at(T, idx[:, g], 2 * coef[:, g, None] * e)
        np.add.at(n, idx[:, g], 1)
    tol = lr * 2.0 ** -24 * ((s + 2) * S + (n[:, None] + 2) * T) + 4e-7
    assert np.all(np.abs(Dd.cpu().numpy() - want_D) <= tol)
    # a scatter to the wrong atom would show: nearly every atom moves by far more than that
    assert np.mean(np.abs(want_D - D0).max(1) > 20 * tol.max(1)) > 0.9
    assert losses[0] == pytest.approx(l_mse, rel=(s + 8) * 2.0 ** -22 * float((A * A).sum() / max(l_mse, 1e-30)) ** 0.5)
    assert losses[1] == pytest.approx(l_div, rel=2e-5)
