"""The time ordering as a matrix product, against the oracle's transforms at the edges of its tiles (128
points, up to 52 times per parity, 16 terms per stage), for point counts that are and are not a multiple of 4."""
import numpy as np
import pytest

from oracle import sgw as osgw
from paper_2601_21005_gb300 import build

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


def _abs_matrix(n):
    """|G(t, j)| of Im u(t) = sum_j G(t, j) u^R(t_j) (zero for equal parities)."""
    M = osgw.time_order_length(n)
    t = np.arange(n + 1)
    g = np.zeros((n + 1, n + 1))
    odd = (t[:, None] + t[None, :]) % 2 == 1
    s, d = (t[:, None] + t[None, :])[odd], (t[:, None] - t[None, :])[odd]
    g[odd] = (1 / np.tan(np.pi * s / M) - 1 / np.tan(np.pi * d / M)) / M
    return np.abs(g)


@pytest.mark.parametrize('n,points', [(0, 5), (1, 64), (2, 63), (3, 1), (15, 66), (16, 65), (31, 128), (63, 7), (103, 127),
                                      (104, 129), (111, 68), (206, 130), (207, 64), (208, 61), (400, 193), (401, 192), (513, 64), (1023, 67)])
def test_time_order_matrix_product(n, points):
    assert torch.cuda.is_available()
    build.build()
    from paper_2601_21005_gb300 import sgw
    r = np.random.default_rng(n)
    x = r.normal(size=(2, n + 1, points)).astype(np.float32)
    c = sgw.Context(16, 0.5)
    u = torch.full((2, n + 1, points), float('nan'), dtype=torch.complex64, device='cuda')
    xd = torch.as_tensor(x).cuda()
    c.time_order_points(xd, u, 2, n, points)
    got = u.cpu().numpy()
    A = _abs_matrix(n)
    for s in range(2):
        ref = osgw.time_order(x[s].astype(np.float64))
        # a chunk of up to 32 terms, up to 17 chunk totals, G itself and the store: at most 52 roundings
        # of 2^-24 on the sum of the magnitudes; the real part is x or x / 2 exactly
        bound = 52 * 2.0 ** -24 * (A @ np.abs(x[s].astype(np.float64))) + 1e-30
        assert np.all(np.abs(got[s].imag - ref.imag) <= bound + 1e-12)
        assert np.all(np.abs(got[s].real - ref.real) <= 1e-12 * np.max(np.abs(x)))
    u2 = torch.empty_like(u)
    c.time_order_points(xd, u2, 2, n, points)                 # the kept matrix gives the same bits
    assert torch.equal(u, u2)


def test_many_step_counts_in_one_context():
    """More step counts than matrices are kept, and back to the first."""
    build.build()
    from paper_2601_21005_gb300 import sgw
    c = sgw.Context(16, 0.5)
    x = torch.randn(1, 41, 70, device='cuda')
    first = None
    for n in list(range(20, 41)) + [20]:
        u = torch.empty(1, n + 1, 70, dtype=torch.complex64, device='cuda')
        c.time_order_points(x[:, :n + 1].contiguous(), u, 1, n, 70)
        if n == 20:
            if first is not None:
                assert torch.equal(u, first)
            first = u


def test_captured_orderings_outlive_other_step_counts():
    """A caller's graph keeps the matrix it was captured with, whatever the context orders afterwards; and the
    step count in constant use stays among those kept."""
    build.build()
    from paper_2601_21005_gb300 import sgw
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        c = sgw.Context(16, 0.5, stream=st.cuda_stream)
        x = torch.randn(1, 61, 70, device='cuda')
        order = lambda n, u: c.time_order_points(x[:, :n + 1].contiguous(), u, 1, n, 70)
        out = lambda n: torch.empty(1, n + 1, 70, dtype=torch.complex64, device='cuda')
        xs = x[:, :21].contiguous()
        u, want = out(20), out(20)
        c.time_order_points(xs, want, 1, 20, 70)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            c.time_order_points(xs, u, 1, 20, 70)
        junk = []
        for n in range(21, 45):
            order(n, out(n))
            order(50, out(50))
            junk.append(torch.full((1 << 18,), float('nan'), device='cuda'))    # would land in memory given back
        g.replay()
    st.synchronize()
    assert torch.equal(u, want)


@pytest.mark.parametrize('kept,captured', [(8, 12), (64, 100), (300, 400), (16, 31)])
def test_step_counts_of_one_length_share_a_capture(kept, captured):
    """A first ordering of one step count lets a capture record any other of the same padded length
    (64, 512, 2048, 128 here), with the bits that the step count's own matrix gives."""
    build.build()
    from paper_2601_21005_gb300 import sgw
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        c = sgw.Context(16, 0.5, stream=st.cuda_stream)
        x = torch.randn(1, captured + 1, 70, device='cuda')
        u = [torch.empty(1, captured + 1, 70, dtype=torch.complex64, device='cuda') for _ in range(2)]
        c.time_order_points(x[:, :kept + 1].contiguous(), u[0][:, :kept + 1].contiguous(), 1, kept, 70)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            c.time_order_points(x, u[0], 1, captured, 70)
        g.replay()
        c.time_order_points(x, u[1], 1, captured, 70)
    st.synchronize()
    assert torch.equal(u[0], u[1])


@pytest.mark.parametrize('n,points', [(50, 1), (63, 127), (79, 300), (103, 1000), (206, 999), (400, 1024), (401, 1001),
                                      (1000, 384)])
def test_few_points_give_the_bits_of_many(n, points):
    """Calls of few points give a tile's rows to several blocks (odd and even numbers of rows to a warp here); a
    point's sums have the same order either way."""
    build.build()
    from paper_2601_21005_gb300 import sgw
    c = sgw.Context(16, 0.5)
    many = 40000
    x = torch.randn(1, n + 1, many, device='cuda')
    u = torch.empty(1, n + 1, many, dtype=torch.complex64, device='cuda')
    c.time_order_points(x, u, 1, n, many)
    few = torch.full((1, n + 1, points), float('nan'), dtype=torch.complex64, device='cuda')
    c.time_order_points(x[..., :points].contiguous(), few, 1, n, points)
    assert torch.equal(few, u[..., :points])
