"""Sums behind Sigma(t) and the QP solve, at the sizes and ranges where their paths change.

Sigma at t = 0 is dV/2 times the difference of two sums of phi zeta u, so with u given it tests the
accumulation alone.  A sum of products of three rounded to FP64 as it goes has at most 2 roundings of
2^-53 in a product and, through thread, warp, block and grid, some 40 additions: 64 * 2^-53 of the sum of
the terms' magnitudes bounds it.  The FP32 form: 2^-24 in place of 2^-53."""
import numpy as np
import pytest

from oracle import sgw as osgw
from paper_2601_21005_gb300 import build

import gpu_common as gc

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


def _ctx(n, batch):
    assert torch.cuda.is_available()
    build.build()
    from paper_2601_21005_gb300 import sgw
    c = sgw.Context(n, 0.5, max_batch=batch)
    c.set_potential(torch.zeros(n ** 3, dtype=torch.float32, device='cuda'), [])
    c.set_spectrum(-1.0, 80.0)
    return c


@pytest.mark.parametrize('n,scale,spread,fp64,zscale', [
    (16, 1.0, 0.0, 1, 1.0), (64, 1.0, 0.0, 1, 1.0),
    (32, 1.0, 12.0, 1, 1.0),              # magnitudes over 24 decades, as in a cluster's tails
    (32, 2.0 ** -110, 0.0, 1, 1.0),       # products below what FP32 halves hold exactly
    (32, 2.0 ** -100, 6.0, 1, 1.0),       # some threads on either side of that line
    (32, 2.0 ** 110, 0.0, 1, 1.0),        # products beyond FP32
    (48, 1.0, 4.0, 0, 1.0),
    (32, 2.0 ** -120, 0.0, 1, 2.0 ** 40),     # products well in range, of factors u phi that are not
    (32, 2.0 ** -130, 0.0, 1, 2.0 ** 60),     # and of subnormal u
    (32, 2.0 ** -85, 3.0, 1, 2.0 ** 12),      # blocks on either side of the line for zeta
])
def test_sums_against_wide_arithmetic(n, scale, spread, fp64, zscale):
    ns, steps, ng = 2, 1, n ** 3
    rng = np.random.default_rng(n + int(spread))
    mag = 10.0 ** (spread * (rng.random(ng) - 0.5) * 2)
    phi = (rng.normal(size=ng) * mag).astype(np.float32)
    u = (scale * (rng.normal(size=(ns, steps + 1, ng)) + 1j * rng.normal(size=(ns, steps + 1, ng)))).astype(np.complex64)
    z = (zscale * (rng.normal(size=(ns, 2, ng)) + 1j * rng.normal(size=(ns, 2, ng)))).astype(np.complex64)
    sig = torch.empty(ns, 2 * steps + 1, dtype=torch.complex128, device='cuda')
    c = _ctx(n, 2 * ns)
    c.sigma_c(gc.to_dev(z, torch, torch.complex64), gc.to_dev(phi, torch, torch.float32),
              gc.to_dev(u, torch, torch.complex64), ns, steps, 0.05, 8, sig, fp64)
    got = sig.cpu().numpy()[:, steps]
    eps = 2.0 ** -53 if fp64 else 2.0 ** -24
    wide = np.longdouble
    for s in range(ns):
        d = z[s, 1].astype(np.clongdouble), z[s, 0].astype(np.clongdouble)
        fu = phi.astype(wide) * u[s, 0].astype(np.clongdouble)
        want = 0.5 * (0.125 * np.sum(d[0] * fu) - 0.125 * np.sum(d[1] * fu))
        size = 0.125 * np.sum((np.abs(d[0]) + np.abs(d[1])) * np.abs(fu))
        assert abs(complex(got[s]) - complex(want)) <= 64 * eps * float(size)


def test_one_point_keeps_fp64_precision():
    """With one point in the grid a sum is a single complex product of three.  FP64 rounds each part of it four
    times at most (u phi is exact): 2 * 2^-53 of its terms' magnitudes, and dV and the halving are exact."""
    n, ns = 16, 64
    ng = n ** 3
    rng = np.random.default_rng(7)
    c = _ctx(n, 2 * ns)
    for _ in range(8):
        at = rng.integers(0, ng, ns)
        z, u = (rng.normal(size=(ns, 2)).astype(np.float32) for _ in range(2))
        phi = rng.normal(size=ng).astype(np.float32)
        f = phi[at]
        zd = np.zeros((ns, 2, ng), np.complex64)
        ud = np.zeros((ns, 1, ng), np.complex64)
        zd[np.arange(ns), 1, at] = z[:, 0] + 1j * z[:, 1]
        ud[np.arange(ns), 0, at] = u[:, 0] + 1j * u[:, 1]
        sig = torch.empty(ns, 1, dtype=torch.complex128, device='cuda')
        c.sigma_c(gc.to_dev(zd, torch, torch.complex64), gc.to_dev(phi, torch, torch.float32),
                  gc.to_dev(ud, torch, torch.complex64), ns, 0, 0.05, 8, sig, 1)
        got = sig.cpu().numpy()[:, 0]
        zl, ul, fl = z.astype(np.longdouble), u.astype(np.longdouble), f.astype(np.longdouble)
        re, im = [zl[:, 0] * fl * ul[:, 0], -zl[:, 1] * fl * ul[:, 1]], [zl[:, 0] * fl * ul[:, 1], zl[:, 1] * fl * ul[:, 0]]
        for part, (a, b) in ((got.real, re), (got.imag, im)):
            assert np.all(np.abs(part - (a + b) / 16) <= 2 * 2.0 ** -53 * (np.abs(a) + np.abs(b)) / 16)


def test_sums_pass_infinities_and_nan_on():
    n, ng = 16, 16 ** 3
    c = _ctx(n, 2)
    one = lambda *s: torch.ones(*s, dtype=torch.complex64, device='cuda')
    phi = torch.ones(ng, dtype=torch.float32, device='cuda')
    sig = torch.empty(1, 3, dtype=torch.complex128, device='cuda')
    for bad in (float('inf'), float('nan')):
        u = one(1, 2, ng)
        u[0, 0, 5] = bad
        c.sigma_c(one(1, 2, ng), phi, u, 1, 1, 0.05, 8, sig, 1)
        assert not np.isfinite(sig.cpu().numpy()[0, 1])
    u = one(1, 2, ng) * 0
    c.sigma_c(one(1, 2, ng), phi, u, 1, 1, 0.05, 8, sig, 1)
    assert sig.cpu().numpy()[0, 1] == 0


@pytest.mark.parametrize('n_s,steps,window', [(1, 3, 2.0), (2, 12, 2.0), (9, 130, 1.0), (41, 500, 0.1), (3, 12, 1e-3)])
def test_qp_solve_against_oracle(n_s, steps, window):
    """A root is a bisection to 1e-10 of the same function: 1e-9, as for the longer-standing QP test."""
    rng = np.random.default_rng(steps)
    dt = 0.05
    gamma = 3.0 / (steps * dt)
    t = dt * np.arange(-steps, steps + 1)
    S = np.array([-0.02j * (1 + 0.3 * rng.normal()) * np.exp(-0.3j * t) * (t > 0)
                  + 0.02j * (1 + 0.3 * rng.normal()) * np.exp(0.4j * t) * (t < 0) for _ in range(n_s)])
    X = (0.0 if window < 1 else -0.05) + 0.01 * rng.normal(size=n_s)
    c = _ctx(16, 2)
    solve = lambda x: c.qp_energy(gc.to_dev(S, torch, torch.complex128), gc.to_dev(x, torch, torch.float64), n_s, steps,
                                  dt, gamma, -0.25, 0.01, window, 1e-3, 1)
    if window == 1e-3:               # two scan steps, and no sign change in them
        from paper_2601_21005_gb300 import sgw
        with pytest.raises(sgw.SgwError):
            solve(X + 5.0)
        return
    r = solve(X)
    e, se = osgw.qp_energy(list(S), list(X), dt, gamma, -0.25, 0.01)
    assert abs(r['eps_qp'] - e) < 1e-9
    assert n_s == 1 or abs(r['se'] - se) < 1e-9
