"""16-bit products of 65 columns or more, over long reductions by SM pairs (256 x 256 tiles, 128 rows per CTA): parity
with the FP64 oracle on the dequantised kernel at the tiles' edges, and the bounded waits.

Tolerance: the spectra are rounded to the 16-bit type after a power-of-two scale, relative error per entry
at most u (2^-11 float16, 2^-8 bfloat16), independent over the sum: u / sqrt(3) expected, 4 u allowed (as
for the narrower tiles).
"""
import numpy as np
import pytest

from oracle import mdc as omdc
from test_gpu_precision import FORMATS, dequantised, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (nr, ns, nf, nv): row tiles exact (256), half used (a whole CTA past the end), one over and one under in
# both directions; one and several column tiles with remainders; one reduction slice and many
CASES = [(256, 128, 3, 128), (100, 60, 4, 65), (257, 129, 3, 127), (255, 127, 3, 130), (129, 400, 2, 256),
         (700, 33, 2, 70)]
# the same edges with a reduction of 20 stages or more, which pairs take: forward, then adjoint
LONG = [(256, 600, 3, 128), (100, 620, 4, 65), (257, 577, 3, 127), (255, 700, 3, 130), (129, 900, 2, 256),
        (1217, 64, 3, 128), (1281, 60, 4, 65), (1300, 129, 3, 127), (1250, 127, 3, 130), (1400, 33, 2, 70)]


def problem(nr, ns, nf, nv, nt=64):
    rng = np.random.default_rng(nr + 7 * ns + 31 * nv)
    G = (rng.standard_normal((nf, nr, ns)) + 1j * rng.standard_normal((nf, nr, ns))) / np.sqrt(ns)
    return G, rng.standard_normal((nt, ns, nv)).astype(np.float32), rng.standard_normal((nt, nr, nv)).astype(np.float32)


@pytest.mark.parametrize("storage", ["c16f", "cbf16"])
@pytest.mark.parametrize("nr,ns,nf,nv", CASES + LONG)
def test_pair_products_match_oracle(storage, nr, ns, nf, nv):
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, nf, nv)
    op = m.MDC(torch.from_numpy(G.astype(np.complex64)).cuda(), 64, 0.004, 400.0, storage=storage)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    m.mdc_device_status(op.h)
    assert m.mdc_tc_fallback_count(op.h) == 0
    op.close()
    Gq = dequantised(G, storage)
    tol = 4 * FORMATS[storage][0]
    assert rel(yg, omdc.forward(Gq, x, 0.004, 400.0)) <= tol
    assert rel(xg, omdc.adjoint(Gq, y, 0.004, 400.0)) <= tol


@pytest.mark.parametrize("storage", ["c16f", "cbf16"])
@pytest.mark.parametrize("nr,ns,nf,nv", [(39, 173, 39, 245), (300, 90, 80, 70), (128, 64, 160, 66)])
def test_single_cta_products_match_oracle(storage, nr, ns, nf, nv):
    """Shapes that pairs would waste (one row tile, three, with a last wave to spare), in one direction or both."""
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, nf, nv, nt=512)
    op = m.MDC(torch.from_numpy(G.astype(np.complex64)).cuda(), 512, 0.004, 400.0, storage=storage)
    yg = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    xg = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    m.mdc_device_status(op.h)
    assert m.mdc_tc_fallback_count(op.h) == 0
    op.close()
    Gq = dequantised(G, storage)
    tol = 4 * FORMATS[storage][0]
    assert rel(yg, omdc.forward(Gq, x, 0.004, 400.0)) <= tol
    assert rel(xg, omdc.adjoint(Gq, y, 0.004, 400.0)) <= tol


def test_pair_wait_limit():
    """A limit the pipeline cannot meet is reported, and the handle works again with the default one."""
    import paper_2011_11120_gb300 as m
    G, x, _ = problem(300, 1100, 20, 100)
    op = m.MDC(torch.from_numpy(G.astype(np.complex64)).cuda(), 64, 0.004, 400.0, storage="c16f")
    xt = torch.from_numpy(x).cuda()
    op.forward(xt)
    m.mdc_device_status(op.h)
    m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, 1)
    for _ in range(5):
        op.forward(xt)
    with pytest.raises(m.MDCError) as e:
        m.mdc_device_status(op.h)
    assert e.value.status == -4
    m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, 0)
    yg = op.forward(xt).cpu().numpy()
    m.mdc_device_status(op.h)
    op.close()
    assert rel(yg, omdc.forward(dequantised(G, "c16f"), x, 0.004, 400.0)) <= 4 * FORMATS["c16f"][0]


@pytest.mark.parametrize("nr,ns", [(300, 1100), (700, 2300), (2300, 400)])
def test_pair_leaves_nothing_behind(nr, ns):
    """Limits around the time of a step, so that waits run out in some pairs and in either CTA of a pair, at any
    step: every launch ends, its status is a timeout or none, and products launched right behind it on the
    same SMs are right."""
    import paper_2011_11120_gb300 as m
    G, x, y = problem(nr, ns, 20, 100)
    op = m.MDC(torch.from_numpy(G.astype(np.complex64)).cuda(), 64, 0.004, 400.0, storage="c16f")
    xt, yt = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    Gq = dequantised(G, "c16f")
    want_y, want_x = omdc.forward(Gq, x, 0.004, 400.0), omdc.adjoint(Gq, y, 0.004, 400.0)
    expired = 0
    for us in (1, 2, 3, 5, 8, 12, 20, 30):
        m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, us)
        for _ in range(3):
            op.forward(xt)
            op.adjoint(yt)
        m.mdc_set_option(op.h, m.MDC_OPT_WAIT_LIMIT_US, 0)
        yg, xg = op.forward(xt).cpu().numpy(), op.adjoint(yt).cpu().numpy()
        try:
            m.mdc_device_status(op.h)
        except m.MDCError as e:
            assert e.status == -4
            expired += 1
        assert rel(yg, want_y) <= 4 * FORMATS["c16f"][0]
        assert rel(xg, want_x) <= 4 * FORMATS["c16f"][0]
    assert expired > 0
    op.close()
