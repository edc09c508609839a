"""Complex64 products on tensor cores (five columns or more): parity with the FP64 oracle at the edges
of the kernel's tiles, and the bounded waits.

Tolerance: each output sums at most 32 chunk sums per group in float32 (RMS rounding 2^-24 / sqrt(3) per
addition against partial sums that grow like a random walk: sqrt(32 / 2) 2^-24 / sqrt(3) = 1.4e-7), each
chunk truncated at most four times by 2^-25 of its size (1.2e-7), between two transforms of about
1.2e-7 each: 2.6e-7 together, and four times that for structure in the data.
"""
import numpy as np
import pytest

from oracle import mdc as omdc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-6

# (nr, ns, nf, nv): column tiles of 32, 64, 96 and 128 real columns with remainders and more than one
# tile; row tiles of 128 kernel rows (64 columns, adjoint) exact, one over, one under; reduction steps of
# 32 reals exact and with a tail, one step, and more than one group of 64 steps in either direction
CASES = [(1, 7, 3, 5), (129, 65, 9, 16), (128, 64, 5, 17), (127, 63, 5, 32), (77, 1100, 6, 33),
         (2100, 40, 5, 48), (130, 129, 4, 49), (64, 50, 4, 64), (33, 300, 4, 65), (200, 31, 3, 130)]


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def problem(nr, ns, nf, nv, nt=64):
    rng = np.random.default_rng(nr + 7 * ns + 31 * nv)
    G = (rng.standard_normal((nf, nr, ns)) + 1j * rng.standard_normal((nf, nr, ns))) / np.sqrt(ns)
    G = G.astype(np.complex64)
    x = rng.standard_normal((nt, ns, nv)).astype(np.float32)
    y = rng.standard_normal((nt, nr, nv)).astype(np.float32)
    return G, x, y


@pytest.mark.parametrize("nr,ns,nf,nv", CASES)
def test_c64_tensor_core_products_match_oracle(nr, ns, nf, nv):
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, nf, nv)
    op = m.MDC(torch.from_numpy(G).cuda(), 64, 0.004, 400.0)
    m.mdc_timing(op.h, True)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    assert m.mdc_timing_read(op.h, "tc_prep")[1] == 2          # both products ran on tensor cores
    yc = op.forward(torch.from_numpy(x).cuda(), conj=True).cpu().numpy()
    m.mdc_device_status(op.h)
    op.close()
    G = G.astype(np.complex128)
    assert rel(yg, omdc.forward(G, x, 0.004, 400.0)) <= TOL
    assert rel(xg, omdc.adjoint(G, y, 0.004, 400.0)) <= TOL
    assert rel(yc, omdc.forward_conj_kernel(G, x, 0.004, 400.0)) <= TOL


@pytest.mark.parametrize("scale", [2.0 ** -100, 1.0, 2.0 ** 100])
@pytest.mark.parametrize("nr,ns,nv", [(40, 2100, 16), (2100, 40, 40)])
def test_sums_of_one_sign_and_range(nr, ns, nv, scale):
    """Real parts of one sign, so that the accumulators' truncation does not cancel, with kernels near either
    end of the range.  Each chunk loses at most four times 2^-25 of itself (1.2e-7), and the float32 additions of
    66 chunk sums at most half an ulp of the running sum each, 2^-25 on average and of either sign: within TOL."""
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, 4, nv)
    G = ((np.abs(G.real) - 1j * np.abs(G.imag)) * scale).astype(np.complex64)
    x, y = (np.abs(x) / scale).astype(np.float32), (np.abs(y) / scale).astype(np.float32)
    op = m.MDC(torch.from_numpy(G).cuda(), 64, 0.004, 400.0)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    op.close()
    G = G.astype(np.complex128)
    assert rel(yg, omdc.forward(G, x, 0.004, 400.0)) <= TOL
    assert rel(xg, omdc.adjoint(G, y, 0.004, 400.0)) <= TOL


def test_c64_tensor_core_wait_limit():
    """A limit the pipeline cannot meet is reported, and the handle works again with the default one.  The kernel
    (0.9 GB) streams from memory: with every SM's ring of loads in flight a tile takes some microseconds."""
    import paper_2011_11120_gb300 as m
    g = torch.Generator(device="cuda").manual_seed(5)
    G = torch.view_as_complex(torch.randn((50, 1024, 2200, 2), generator=g, device="cuda"))
    op = m.MDC(G, 128, 0.004, 400.0)
    xt = torch.randn((128, 2200, 16), generator=g, device="cuda")
    want = op.forward(xt)
    m.mdc_device_status(op.h)
    m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, 1)
    for _ in range(40):
        op.forward(xt)
    with pytest.raises(m.MDCError) as e:
        m.mdc_device_status(op.h)
    assert e.value.status == -4
    m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, 0)
    yg = op.forward(xt)
    m.mdc_device_status(op.h)
    op.close()
    assert torch.equal(yg, want)


@pytest.mark.parametrize("nv", [3, 9])
def test_marchenko_products_stay_in_float32(nv):
    """A solve's complex64 products run on the float32 kernels, whether or not the handle holds the operand
    that passes of as many columns use: the same bits either way."""
    import paper_2011_11120_gb300 as m
    nt, n, nf = 128, 70, 20
    rng = np.random.default_rng(nv)
    G = (rng.standard_normal((nf, n, n)) + 1j * rng.standard_normal((nf, n, n))) * (0.2 / np.sqrt(n))
    cut = torch.from_numpy(rng.integers(nt // 16, nt // 2, (n, nv)).astype(np.int32)).cuda()
    fd = torch.from_numpy(rng.standard_normal((nt, n, nv)).astype(np.float32)).cuda()
    got = []
    for reserve in (False, True):
        op = m.MDC(torch.from_numpy(G.astype(np.complex64)).cuda(), nt, 1.0, 1.0)
        if reserve:
            m.mdc_reserve(op.h, 2 * nv)
        m.mdc_timing(op.h, True)
        out, neu = op.marchenko(cut, fd, 3), op.neumann(cut, fd, 3)
        assert m.mdc_timing_read(op.h, "tc_prep")[1] == 0
        op.forward(fd.repeat(1, 1, 2))
        assert m.mdc_timing_read(op.h, "tc_prep")[1] == 1          # a pass of 2 nv columns does use it
        got.append([t[k].cpu().numpy() for t in (out, neu) for k in ("f_minus", "f_mplus", "g_minus", "g_plus")])
        op.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_operand_limit():
    """A smaller operand takes wide products in slabs with the same bits; none at all sends them to the float32
    kernels, counted, until a call finds room again."""
    import paper_2011_11120_gb300 as m
    G, x, y = problem(333, 700, 8, 200)
    op = m.MDC(torch.from_numpy(G).cuda(), 64, 0.004, 400.0)
    xt, yt = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()

    def both():
        m.mdc_timing(op.h, True)
        out = op.forward(xt).cpu().numpy(), op.adjoint(yt).cpu().numpy()
        return out, m.mdc_timing_read(op.h, "tc_prep")[1], m.mdc_tc_fallback_count(op.h)

    full, preps, count = both()
    assert (preps, count) == (2, 0)
    m.mdc_set_option(op.h, m.MDC_OPT_C64_OPERAND_MB, 9)           # 69 of 200 columns: slabs of a 64-column tile
    slabs, preps, count = both()
    assert (preps, count) == (8, 0)
    m.mdc_set_option(op.h, m.MDC_OPT_C64_OPERAND_MB, 1)
    none, preps, count = both()
    assert (preps, count) == (0, 2)
    m.mdc_set_option(op.h, m.MDC_OPT_C64_OPERAND_MB, 0)
    again, preps, count = both()
    assert (preps, count) == (2, 2)
    m.mdc_device_status(op.h)
    op.close()
    G = G.astype(np.complex128)
    want = omdc.forward(G, x, 0.004, 400.0), omdc.adjoint(G, y, 0.004, 400.0)
    for f, s, n, a, w in zip(full, slabs, none, again, want):
        assert np.array_equal(f, s) and np.array_equal(f, a)
        assert rel(f, w) <= TOL and rel(n, w) <= TOL


@pytest.mark.parametrize("ncol", [20, 40])
def test_float32_gemm_matches_oracle(ncol):
    """The SIMT GEMM's narrow and wide tiles, which products without the operand run on, in both directions."""
    import paper_2011_11120_gb300 as m
    G, x, y = problem(131, 497, 9, ncol)
    op = m.MDC(torch.from_numpy(G).cuda(), 64, 0.004, 400.0)
    m.mdc_set_option(op.h, m.MDC_OPT_C64_OPERAND_MB, 1)           # the operand takes 110 KB a column
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    used = m.mdc_tc_fallback_count(op.h)
    op.close()
    G = G.astype(np.complex128)
    assert rel(yg, omdc.forward(G, x, 0.004, 400.0)) <= TOL
    assert rel(xg, omdc.adjoint(G, y, 0.004, 400.0)) <= TOL
    assert used == 2


# (nr, ns, nv, products on tensor cores): either side of the bounds of the smallest kernels
@pytest.mark.parametrize("nr,ns,nv,preps", [(32, 32, 5, 0), (33, 32, 24, 2), (32, 32, 33, 2), (160, 204, 8, 1), (161, 204, 8, 2),
                                            (160, 205, 8, 2), (100, 100, 9, 2), (30, 1000, 17, 1), (30, 1000, 16, 2)])
def test_smallest_kernels_match_oracle(nr, ns, nv, preps):
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, 5, nv)
    op = m.MDC(torch.from_numpy(G).cuda(), 64, 0.004, 400.0)
    m.mdc_timing(op.h, True)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    got = m.mdc_timing_read(op.h, "tc_prep")[1], m.mdc_tc_fallback_count(op.h)
    op.close()
    G = G.astype(np.complex128)
    assert rel(yg, omdc.forward(G, x, 0.004, 400.0)) <= TOL
    assert rel(xg, omdc.adjoint(G, y, 0.004, 400.0)) <= TOL
    assert got == (preps, 0)
