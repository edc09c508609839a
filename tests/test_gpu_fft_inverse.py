"""Inverse transforms (spectrum read straight into registers) and the forward transforms of odd column
counts: every length, even and odd columns, few-column and full tiles, bands of one bin, of part of the
lower blocks and of the whole spectrum (DC and Nyquist), alone and with the fused solver epilogue.

Tolerance: float32 transforms of log2(nt) <= 10 stages and short sums, relative 2-norm about 2e-7 per
pass; 1e-6 for a pass, 1e-5 for a solve (as the solver tests).
"""
import numpy as np
import pytest

from oracle import marchenko as omar
from oracle import mdc as omdc
from oracle import solvers

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def kernel(n, m, nf, seed):
    rng = np.random.default_rng(seed)
    G = (rng.standard_normal((nf, n, m)) + 1j * rng.standard_normal((nf, n, m))).astype(np.complex64)
    return rng, G * np.float32(0.2 / np.sqrt(max(n, m)))


# columns: 7 x 3 = 21 (odd, few), 10 x 4 = 40, 911 x 5 = 4555 (odd, full tiles), 700 x 8 = 5600
@pytest.mark.parametrize("nt", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("n,nv", [(7, 3), (10, 4), (911, 5), (700, 8)])
@pytest.mark.parametrize("band", ["one", "part", "all"])
def test_pass_matches_oracle(nt, n, nv, band):
    import paper_2011_11120_gb300 as m
    nf = {"one": 1, "part": nt // 5, "all": nt // 2 + 1}[band]
    if n > 100 and band == "all":
        nf, n, nv = nt // 2 + 1, n // 30, nv * 30 + n % 2         # the same column range, a small kernel
    rng, G = kernel(n, 6, nf, nt + n + nv + nf)
    x = rng.standard_normal((nt, 6, nv)).astype(np.float32)
    y = rng.standard_normal((nt, n, nv)).astype(np.float32)
    op = m.MDC(torch.from_numpy(G).cuda(), nt, 1.0, 1.0)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda(), conj=True).cpu().numpy()
    op.close()
    G = G.astype(np.complex128)
    assert rel(yg, omdc.forward(G, x, 1.0, 1.0)) <= 1e-6
    assert rel(xg, omdc.adjoint_conj_kernel(G, y, 1.0, 1.0)) <= 1e-6


@pytest.mark.parametrize("nt", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("n,nv", [(7, 3), (6, 4), (61, 61)])
def test_solver_epilogue_matches_oracle(nt, n, nv):
    import paper_2011_11120_gb300 as m
    nf = nt // 4
    rng, G = kernel(n, n, nf, nt + n)
    cut = rng.integers(nt // 16, nt // 2, (n, nv)).astype(np.int32)
    fd = rng.standard_normal((nt, n, nv)).astype(np.float32)
    op = m.MDC(torch.from_numpy(G).cuda(), nt, 1.0, 1.0)
    out = op.marchenko(torch.from_numpy(cut).cuda(), torch.from_numpy(fd).cuda(), 3)
    op.close()
    ref = omar.Marchenko(G, 1.0, 1.0, cut, nt)
    res = solvers.lsqr(ref.matvec, ref.rmatvec, ref.data(fd), niter=3)
    gm, _, gp = ref.greens(res.x[0], res.x[1], fd)
    for key, want in (("f_minus", res.x[0]), ("f_mplus", res.x[1]), ("g_minus", gm), ("g_plus", gp)):
        assert rel(out[key].cpu().numpy(), want) <= 1e-5, key
    assert np.allclose(out["resid"], res.resid, rtol=1e-5, atol=0)


def chain_norm(d, nt, C):
    """sqrt of the sum of squares of d [nt, C] as the inverse kernels form it: row rho of their tile holds the
    sample t = (rho mod N2) N1 + rho / N2; rows of one column with equal rho mod TS are added up by float32
    fused multiply-adds in ascending order, the chains and the columns in float64."""
    N1, N2, CT = {64: (8, 8, 64), 128: (16, 8, 64), 256: (16, 16, 64), 512: (32, 16, 32), 1024: (32, 32, 16)}[nt]
    TS = (4 if C % 4 == 0 else 1) * 256 // CT
    rho = np.arange(nt)
    rows = d[(rho % N2) * N1 + rho // N2].astype(np.float64)
    ss = np.zeros((TS, C))
    for m in range(nt // TS):
        ss = (rows[m * TS:(m + 1) * TS] ** 2 + ss).astype(np.float32).astype(np.float64)
    return np.sqrt(ss.sum())


@pytest.mark.parametrize("nt", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("n,nv", [(7, 3), (10, 1), (12, 3), (160, 4), (1601, 3)])
def test_norm_does_not_depend_on_the_tile(nt, n, nv):
    """The norm of a solve's data vector (few-column and full tiles) is the sum of the same chains.  Tolerance:
    one chain in a thousand off by a rounding (2^-24), which float64 may take twice here."""
    import paper_2011_11120_gb300 as m
    nf = 6
    rng, G = kernel(n, n, nf, nt + n)
    cut = rng.integers(nt // 16, nt // 2, (n, nv)).astype(np.int32)
    fd = torch.from_numpy(rng.standard_normal((nt, n, nv)).astype(np.float32)).cuda()
    op = m.MDC(torch.from_numpy(G).cuda(), nt, 1.0, 1.0)
    d = op.forward(fd).cpu().numpy().reshape(nt, n * nv)
    resid = op.marchenko(torch.from_numpy(cut).cuda(), fd, 1)["resid"]
    op.close()
    t = np.arange(nt)
    d[np.where(t < nt // 2, t, nt - t)[:, None] >= cut.reshape(1, -1)] = 0.0
    want = chain_norm(d, nt, n * nv)
    assert abs(resid[0] / want - 1.0) <= 1e-10
