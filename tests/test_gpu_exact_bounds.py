"""The exact mode's fp16 sweep knows every correlation to a band that it takes from the norms of its operands' roundings:
the band holds on every pick it decides, and dictionaries whose atoms are far from unit norm get the picks of
fp64 arithmetic too."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def csr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2412_11741_b200 as m
    return m


CHILD = r'''
import sys
import torch
sys.path.insert(0, %(root)r)
import paper_2412_11741_b200 as csr
from paper_2412_11741_b200 import workloads as wl

for engine in (0, 2):
    csr.csr_set_option("exact_engine", engine)
    for w in (wl.dict_sweep(4096, M=8192), wl.dict_sweep(1000, d=64, M=3000), wl.sparsity_sweep(32, tokens=128, N=8192)):
        X = torch.from_numpy(w.X).cuda()
        for scale in (1.0, 3e4, 1e-5):
            D = (torch.from_numpy(w.D).cuda() * scale).contiguous()
            csr.csr_encode_ex(D, X, w.s, mode=csr.CSR_MODE_FP32_EXACT)
            assert csr.csr_device_status() == csr.CSR_OK, csr.csr_last_error_string()
            print("USE", csr.csr_debug_read("exact_band_use"), csr.csr_debug_read("exact_tensor_error"))
'''


def test_the_band_holds_on_every_pick_it_decides():
    """Half the band is a bound (Cauchy-Schwarz on measured norms), so no deviation may use it up; what the tensor cores' own
    sums add stays within its allowance of 2^-15 plus the keys' truncation of 2^-16."""
    from paper_2412_11741_b200 import build
    env = dict(os.environ, CSR_LIBRARY_PATH=build.build(debug=True))
    res = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}], env=env, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout + res.stderr
    lines = [l.split() for l in res.stdout.splitlines() if l.startswith("USE")]
    assert len(lines) == 18
    for _, use, own in lines:
        assert 0.0 < float(use) < 1.0 and float(own) < 2.0 ** -15 + 2.0 ** -16, (use, own)


def _pursuit64(D, X, s):
    D, R = D.double(), X.double()
    idx, coef = [], []
    for _ in range(s):
        corr = R @ D.T
        n = corr.abs().argmax(dim=1)
        c = corr.gather(1, n[:, None])
        R = R - c * D[n]
        idx.append(n)
        coef.append(c)
    return torch.stack(idx, 1), torch.cat(coef, 1)


@pytest.mark.parametrize("engine", [0, 2])
@pytest.mark.parametrize("M,N,d", [(130, 700, 128), (3000, 1500, 64)])
@pytest.mark.parametrize("norms", ["tiny", "huge", "mixed", "one outlier", "first zero"])
def test_dictionaries_of_any_norm_get_the_picks_of_fp64(csr, engine, M, N, d, norms):
    g = torch.Generator(device=DEV).manual_seed(N + len(norms))
    D = torch.nn.functional.normalize(torch.randn(N, d, device=DEV, generator=g), dim=1)
    if norms == "tiny":
        D *= 2.0 ** -40
    elif norms == "huge":
        D *= 2.0 ** 30
    elif norms == "mixed":
        D *= torch.exp(torch.randn(N, 1, device=DEV, generator=g))
    elif norms == "one outlier":                            # beyond fp16 next to the others: every row is searched for in fp64
        D[N // 2 + 1] *= 2.0 ** 20
    else:
        D[: N - 3] = torch.where(torch.arange(N - 3, device=DEV)[:, None] % max(1, N // 32) == 0, torch.zeros_like(D[: N - 3]), D[: N - 3])
    D, X = D.contiguous(), torch.randn(M, d, device=DEV, generator=g)
    s = 1 if norms in ("huge", "one outlier", "mixed") else 4   # (atoms longer than sqrt 2 blow the residual up)
    csr.csr_set_option("exact_engine", engine)
    try:
        idx, coef = csr.csr_encode_ex(D, X, s, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
        assert csr.csr_device_status() == csr.CSR_OK
    finally:
        csr.csr_set_option("exact_engine", 0)
    want_i, want_c = _pursuit64(D, X, s)
    assert torch.equal(idx.view(torch.int16).long() & 0xFFFF, want_i)
    # fp64 sums in two orders, rounded once to fp32
    assert torch.allclose(coef.double(), want_c, rtol=2.0 ** -23, atol=0.0)


@pytest.mark.parametrize("engine", [0, 2])
def test_atoms_that_are_not_finite_are_met_as_they_are(csr, engine):
    """An atom of NaN is never picked and changes nothing about the others."""
    g = torch.Generator(device=DEV).manual_seed(9)
    D = torch.nn.functional.normalize(torch.randn(600, 128, device=DEV, generator=g), dim=1).contiguous()
    X = torch.randn(500, 128, device=DEV, generator=g)
    csr.csr_set_option("exact_engine", engine)
    try:
        keep = csr.csr_encode_ex(torch.cat([D, torch.zeros_like(D[:1])]).contiguous(), X, 4, mode=csr.CSR_MODE_FP32_EXACT)
        got = csr.csr_encode_ex(torch.cat([D, torch.full_like(D[:1], float("nan"))]).contiguous(), X, 4, mode=csr.CSR_MODE_FP32_EXACT)
        assert csr.csr_device_status() == csr.CSR_OK
    finally:
        csr.csr_set_option("exact_engine", 0)
    assert torch.equal(keep[0].view(torch.int16), got[0].view(torch.int16)) and torch.equal(keep[1], got[1])


@pytest.mark.parametrize("engine", [0, 2])
@pytest.mark.parametrize("M,N,d", [(6, 1000, 128), (130, 515, 64), (700, 2100, 128), (3000, 1030, 64)])
@pytest.mark.parametrize("apart", [1, 3, 8, 130])
def test_near_ties_within_and_across_groups(csr, engine, M, N, d, apart):
    """The sweep keeps the largest of eight adjacent atoms: atoms almost alike at the same place of their group, in the same group
    and further apart, closer than the sweep can tell and not closer than fp64 can; exact copies go to the lower one."""
    g = torch.Generator(device=DEV).manual_seed(N + apart)
    D = torch.randn(N, d, device=DEV, generator=g)
    near = torch.arange(16, N - apart, 2 * apart + 17, device=DEV)
    D[near + apart] = D[near] + 10.0 ** torch.empty(len(near), 1, device=DEV).uniform_(-6, -2, generator=g) * torch.randn(len(near), d, device=DEV, generator=g)
    D = torch.nn.functional.normalize(D, dim=1)
    D[9], D[9 + apart] = D[8], -D[8]
    D = D.contiguous()
    pick = near[torch.randint(0, len(near), (M,), device=DEV, generator=g)]
    X = (D[pick] * (1.0 + torch.rand(M, 1, device=DEV, generator=g)) + 0.02 * torch.randn(M, d, device=DEV, generator=g)).contiguous()
    X[0] = -2.0 * D[8]
    csr.csr_set_option("exact_engine", engine)
    try:
        idx, coef = csr.csr_encode_ex(D, X, 3, mode=csr.CSR_MODE_FP32_EXACT, coef_dtype=torch.float32)
        assert csr.csr_device_status() == csr.CSR_OK
    finally:
        csr.csr_set_option("exact_engine", 0)
    got = idx.view(torch.int16).long() & 0xFFFF
    assert int(got[0, 0]) == 8
    Dd, R = D.double(), X.double()
    for k in range(3):                                     # each pick is a largest correlation of fp64's, to fp64's own rounding
        corr = (R @ Dd.T).abs()
        best = corr.max(dim=1).values
        mine = corr.gather(1, got[:, k:k + 1])[:, 0]
        # (a residual is known to 128 roundings of the row: X[0] is a multiple of an atom, what its first pick leaves is nothing else)
        unsure = 128 * 2.0 ** -52 * X.double().norm(dim=1)
        assert bool((best - mine <= unsure).all())
        c = (R * Dd[got[:, k]]).sum(1)
        assert bool(((coef[:, k].double() - c).abs() <= 2.0 ** -22 * c.abs() + unsure).all())
        R = R - c[:, None] * Dd[got[:, k]]
