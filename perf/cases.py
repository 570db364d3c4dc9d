"""Timed cases of the library: the calls a user's program makes, with their inputs.

Every case is one pass through the public Python entry points (`sgw.Context`, `sgw.MLP`,
`pipeline.Pipeline`).  The listed sizes are those of the repository's configurations and tests
(16^3 wells, Si clusters on 32^3 .. 128^3 grids, a large cluster on the 288^3 grid); `draw` gives
more of the same ranges.  `exact` restates each call in 64-bit torch, without the library.
"""
import functools
import math

import numpy as np
import torch

from paper_2601_21005_gb300 import sgw, synth
from paper_2601_21005_gb300.pipeline import Pipeline

DEV = 'cuda'
C64, C128, F32, F64 = torch.complex64, torch.complex128, torch.float32, torch.float64
RADIUS = {32: 4.5, 48: 4.5, 64: 10.5, 96: 14.0, 128: 28.0, 288: 40.0}   # bohr, h = 0.5
LARGEST = 288 ** 3 * 16 * 16             # grid points x vectors x Chebyshev terms of the largest case


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one H psi on the tiny periodic system: a call whose cost is its launches (eigensolvers,
        # the power iteration)
        dict(name='apply_h_16', kind='apply_h', n=16, batch=1),
        # a whole small run through the pipeline with graph replay: noise, filter, exchange, TDH,
        # time ordering, zeta propagation, Sigma(t), and the QP solve
        dict(name='whole_32', kind='whole', n=32, samples=2, group=1, n_eta=3, steps=12, deg=16, n_cheb=96, graphs=True),
        # the TDH response of one sample on a grid whose side is not a power of two
        dict(name='tdh_48', kind='tdh', n=48, samples=1, n_eta=3, steps=3, deg=16),
        # the occupied filter of 4 samples' white noise (9 vectors each); degree cut from 2000
        dict(name='filter_64', kind='filter', n=64, batch=36, n_cheb=200),
        # the TDH propagation of 4 samples x 8 eta pairs, the batch of a production run
        dict(name='tdh_64', kind='tdh', n=64, samples=4, n_eta=8, steps=4, deg=16),
        # the zeta propagation with the Sigma(t) sums of those samples (8 vectors: a small batch)
        dict(name='sigma_64', kind='sigma', n=64, samples=4, steps=12, deg=16, fp64=1),
        # the time ordering of one sample's full-grid u^R over a production run's 400 steps
        dict(name='time_order_64', kind='time_order', points=64 ** 3, samples=1, steps=400),
        # the split-operator stepper, a ragged batch propagated in both directions
        dict(name='split_64', kind='split', n=64, batch=27, steps=10),
        # plain propagation of an odd batch on a radix-3 grid
        dict(name='propagate_96', kind='propagate', n=96, batch=7, steps=2, deg=14),
        # plain propagation on the medium cluster's grid
        dict(name='propagate_128', kind='propagate', n=128, batch=12, steps=1, deg=16),
        # one TDH step of one sample (16 orbitals) of a large cluster, u^R compressed to 10^4 xi functions
        dict(name='tdh_xi_288', kind='tdh_xi', n=288, samples=1, n_eta=8, steps=1, deg=16, n_xi=10000, f_g=0.003, L=32),
        # the control variate's network at the size of a 400-step run: loss and gradients of a
        # mini-batch, then predictions for cheap samples
        dict(name='net_256', kind='net', n_in=148, width=256, n_out=1603, rows=32, cheap=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(['apply_h', 'whole', 'tdh', 'filter', 'sigma', 'time_order', 'split', 'propagate', 'tdh_xi',
                       'net'])
    if kind == 'apply_h':
        n = rng.choice([16, 32, 48, 64, 96, 128])
        return dict(kind=kind, n=n, batch=_log_int(rng, 1, max(1, min(64, 3 * 10 ** 7 // n ** 3))))
    if kind == 'whole':
        n = rng.choice([16, 32, 48])
        return dict(kind=kind, n=n, samples=rng.randint(1, 3), group=rng.randint(1, 2), n_eta=rng.randint(1, 5),
                    steps=_log_int(rng, 3, 24), deg=rng.randint(8, 18), n_cheb=_log_int(rng, 24, 160),
                    graphs=rng.random() < 0.5)
    if kind in ('tdh', 'tdh_xi'):
        n = rng.choice([16, 32, 48, 64, 96, 128] if kind == 'tdh' else [32, 48, 64, 96, 128, 288])
        deg, steps = rng.randint(6, 16), (1 if n == 288 else rng.randint(1, 6))
        room = max(1, min(64, LARGEST // 4 // (n ** 3 * deg * steps))) if n < 288 else 16
        n_eta = min(8, _log_int(rng, 1, max(1, room // 2)))
        c = dict(kind=kind, n=n, samples=rng.randint(1, max(1, min(4, room // (2 * n_eta)))), n_eta=n_eta, steps=steps,
                 deg=deg)
        if kind == 'tdh_xi':
            c.update(n_xi=_log_int(rng, 50, 10000), f_g=rng.choice([0.003, 0.01]), L=rng.choice([32, 16, 8]))
        return c
    if kind in ('filter', 'propagate', 'split'):
        n = rng.choice([16, 32, 64, 128] if kind == 'split' else [16, 32, 48, 64, 96, 128])
        terms = _log_int(rng, 16, 256) if kind == 'filter' else rng.randint(8, 18)
        steps = 1 if kind == 'filter' else rng.randint(1, 8)
        per = n ** 3 * terms * steps
        batch = _log_int(rng, 1, max(1, min(64, LARGEST // 4 // per)))
        if kind == 'filter':
            return dict(kind=kind, n=n, batch=batch, n_cheb=terms)
        if kind == 'propagate':
            return dict(kind=kind, n=n, batch=batch, steps=steps, deg=terms)
        return dict(kind=kind, n=n, batch=batch, steps=steps)
    if kind == 'sigma':
        n = rng.choice([16, 32, 48, 64, 96])
        return dict(kind=kind, n=n, samples=rng.randint(1, 4), steps=rng.randint(1, 8), deg=rng.randint(8, 16),
                    fp64=1)
    if kind == 'time_order':
        steps = _log_int(rng, 3, 1000)
        return dict(kind=kind, points=_log_int(rng, 1000, min(64 ** 3, 10 ** 8 // (steps + 1))), samples=rng.randint(1, 2),
                    steps=steps)
    return dict(kind='net', n_in=rng.choice([20, 64, 148]), width=rng.choice([64, 128, 256]),
                n_out=_log_int(rng, 40, 1603), rows=_log_int(rng, 5, 128), cheap=_log_int(rng, 20, 2000))


# ------------------------------------------------------------------ systems and inputs
@functools.lru_cache(maxsize=None)
def _system(n):
    if n == 16:
        return synth.wells(n=16, h=0.6)
    return synth.si_cluster(n=n, h=0.5, radius=RADIUS[n])


def _spectrum(n):
    """An interval that encloses the spectrum: the wells, the kinetic maximum and the KB energies."""
    s = _system(n)
    return float(s['vloc'].min()) - 1.5, 1.5 * (math.pi / s['h']) ** 2 + 3.0


def _context(n, batch):
    s = _system(n)
    ctx = sgw.Context(n, s['h'], max_batch=batch)
    ctx.set_potential(torch.as_tensor(s['vloc'].reshape(-1).astype(np.float32)).to(DEV), s['kb_atoms'])
    ctx.set_spectrum(*_spectrum(n))
    return ctx


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) + 12345)


def _noise(n, batch, g):
    """Real white noise +-1/sqrt(dV), as the library draws it."""
    amp = _system(n)['h'] ** -1.5
    return (torch.randint(0, 2, (batch, n ** 3), generator=g, device=DEV, dtype=torch.int8).to(F32) * 2 - 1) * amp


def _occupied(n, batch, g):
    """Real low-energy vectors: white noise without the components above 2 Ha (filtered orbitals)."""
    h = _system(n)['h']
    k2 = _k2(n, h, F32)
    out = torch.empty(batch, n ** 3, dtype=C64, device=DEV)
    for b in range(batch):
        f = torch.fft.fftn(_noise(n, 1, g).view(n, n, n)) * torch.exp(-(0.25 * k2) ** 2)
        out[b] = torch.fft.ifftn(f).real.reshape(-1).to(C64)
    return out


def _phi(n):
    s = _system(n)
    c = 0.5 * n * s['h']
    return torch.as_tensor(synth.smooth_orbital(n, s['h'], (c, c, c)).reshape(-1).astype(np.float32)).to(DEV)


def _dirs(batch):
    return np.array([1 if b % 3 else -1 for b in range(batch)], dtype=np.int8)


def _filter_coeffs(case):
    """Jackson-damped Chebyshev coefficients of the step at the occupied edge."""
    lo, hi = _spectrum(case['n'])
    N = case['n_cheb'] + 1
    th = math.acos((-0.1 - 0.5 * (hi + lo)) / (0.5 * (hi - lo)))
    k = np.arange(N)
    a = np.where(k == 0, 1.0 - th / math.pi, -2.0 * np.sin(k * th) / (math.pi * np.maximum(k, 1)))
    q = math.pi / (N + 1)
    return a * ((N - k + 1) * np.cos(q * k) + np.sin(q * k) / np.tan(q)) / (N + 1)


def _inputs(case, seed):
    """The tensors a program has in hand before the call (made from the seed alone)."""
    g, kind = _gen(seed), case['kind']
    if kind in ('apply_h', 'filter'):
        x = _noise(case['n'], case['batch'], g)
        return dict(x=torch.complex(x, torch.zeros_like(x)))
    if kind in ('propagate', 'split'):
        x = _occupied(case['n'], case['batch'], g)
        return dict(x=x * torch.exp(1j * torch.rand(x.shape, generator=g, device=DEV)))
    if kind in ('tdh', 'tdh_xi'):
        n, ns = case['n'], case['samples']
        return dict(eta=_occupied(n, ns * case['n_eta'], g), source=(_noise(n, ns, g) * _phi(n)).contiguous())
    if kind == 'sigma':
        n, ns = case['n'], case['samples']
        occ = _occupied(n, ns, g)
        z = torch.stack([occ, _noise(n, ns, g) - occ], dim=1).reshape(2 * ns, -1).contiguous()
        u = torch.empty(ns, case['steps'] + 1, n ** 3, dtype=C64, device=DEV)
        torch.view_as_real(u).normal_(generator=g).mul_(0.1)
        return dict(z=z, u=u, phi=_phi(n))
    if kind == 'time_order':
        t = torch.arange(case['steps'] + 1, device=DEV, dtype=F32)[None, :, None] * 0.05
        w = torch.rand(case['samples'], 1, case['points'], generator=g, device=DEV) * 3
        a = torch.randn(case['samples'], 1, case['points'], generator=g, device=DEV)
        return dict(uR=(a * torch.sin(w * t) * torch.exp(-0.1 * t)).contiguous())
    if kind == 'net':
        r = lambda *s: torch.randn(*s, generator=g, device=DEV)
        dims = [case['n_in']] + 3 * [case['width']] + [case['n_out']]
        p = []
        for a, b in zip(dims[:-1], dims[1:]):
            p += [(r(a, b) / math.sqrt(a)).reshape(-1), 0.1 * r(b)]
        return dict(x=r(case['rows'], case['n_in']), t=r(case['rows'], case['n_out']), xc=r(case['cheap'], case['n_in']),
                    params=torch.cat(p).cpu().numpy())
    return {}                            # 'whole': the pipeline draws its own noise from the seed


def prepare(case, seed):
    kind, st = case['kind'], _inputs(case, seed)
    st['case'] = case
    if kind == 'whole':
        n, s = case['n'], _system(case['n'])
        st['pl'] = Pipeline(n, s['h'], s['vloc'], s['kb_atoms'], _phi(n).cpu().numpy(), -0.15, -0.05,
                            n_eta=case['n_eta'], n_steps=case['steps'], dt=0.05, cheb_deg=case['deg'],
                            samples_per_batch=case['samples'], seed=int(seed) + 1, stream_id=1,
                            spectrum=_spectrum(n), coeffs=_filter_coeffs(case), graphs=bool(case['graphs']),
                            zeta_group=case['group'])
        ns = case['samples'] * case['group']
        st['sig'] = torch.empty(ns, 2 * case['steps'] + 1, dtype=C128, device=DEV)
        st['xs'] = torch.empty(ns, dtype=F64, device=DEV)
    elif kind == 'net':
        st['net'] = sgw.MLP(case['n_in'], case['width'], case['n_out'], max(case['rows'], case['cheap']), seed=3)
        st['net'].set_params(st['params'])
        st['y'] = torch.empty(case['cheap'], case['n_out'], dtype=F32, device=DEV)
    elif kind == 'time_order':
        st['ctx'] = sgw.Context(16, 0.5, max_batch=1)
        st['u'] = torch.empty(st['uR'].shape, dtype=C64, device=DEV)
    elif kind in ('tdh', 'tdh_xi'):
        st['ctx'] = _context(case['n'], 2 * case['samples'] * case['n_eta'])
        npts = case['n'] ** 3 if kind == 'tdh' else case['n_xi']
        st['uR'] = torch.empty(case['samples'], case['steps'] + 1, npts, dtype=F32, device=DEV)
    elif kind == 'sigma':
        st['ctx'] = _context(case['n'], 2 * case['samples'])
        st['zw'] = torch.empty_like(st['z'])
        st['sig'] = torch.empty(case['samples'], 2 * case['steps'] + 1, dtype=C128, device=DEV)
    else:
        st['ctx'] = _context(case['n'], case['batch'])
        st['out'] = torch.empty_like(st['x'])
        if kind == 'filter':
            st['coeffs'] = _filter_coeffs(case)
    return st


def run(st):
    case = st['case']
    kind, c = case['kind'], st.get('ctx')
    if kind == 'apply_h':
        c.apply_h(st['x'], st['out'])
        return st['out']
    if kind == 'filter':
        c.filter_occupied(st['coeffs'], st['x'], st['out'])
        return st['out']
    if kind == 'propagate':              # in place: the program keeps its start vectors
        st['out'].copy_(st['x'])
        c.propagate(st['out'], case['steps'], 0.05, case['deg'], _dirs(case['batch']))
        return st['out']
    if kind == 'split':
        st['out'].copy_(st['x'])
        c.propagate_split(st['out'], case['steps'], 0.05, _dirs(case['batch']))
        return st['out']
    if kind == 'tdh':
        c.tdh_response(st['eta'], st['source'], case['samples'], case['n_eta'], case['steps'], 0.05, case['deg'],
                       st['uR'])
        return st['uR']
    if kind == 'tdh_xi':
        c.tdh_response_xi(st['eta'], st['source'], case['samples'], case['n_eta'], case['steps'], 0.05, case['deg'],
                          _xi(case), st['uR'])
        return st['uR']
    if kind == 'sigma':
        st['zw'].copy_(st['z'])
        c.sigma_c(st['zw'], st['phi'], st['u'], case['samples'], case['steps'], 0.05, case['deg'], st['sig'],
                  case['fp64'])
        return dict(sigma=st['sig'], zeta=st['zw'])
    if kind == 'time_order':
        c.time_order_points(st['uR'], st['u'], case['samples'], case['steps'], case['points'])
        return st['u']
    if kind == 'whole':
        pl = st['pl']
        pl.run_batch(0, st['sig'], st['xs'])
        r = pl.qp(st['sig'], st['xs'], -0.15)
        return dict(sigma=st['sig'], x=st['xs'], eps_qp=r['eps_qp'])
    loss, grads = st['net'].gradients(st['x'], st['t'], want_grads=True)
    st['net'].forward(st['xc'], st['y'])
    return dict(loss=loss, grads=grads, y=st['y'])


def _xi(case):
    return (77, 5, 0, case['n_xi'], case['f_g'], case['L'])


# ------------------------------------------------------------------ compulsory work and tolerances
def _series(ng, vectors, terms):
    """Operations of `terms` H applications and recurrence updates: an FFT pair and about 30 more."""
    return ng * vectors * terms * (10 * math.log2(ng) + 30)


def work(case):
    """Inputs read once, outputs written once; operations of the method's transforms and products."""
    kind = case['kind']
    ng = case.get('n', 0) ** 3
    v4 = 4 * ng
    if kind in ('apply_h', 'filter', 'propagate', 'split'):
        b = case['batch']
        terms = {'apply_h': 1, 'filter': case.get('n_cheb'), 'split': case.get('steps')}.get(kind)
        if kind == 'propagate':
            terms = case['steps'] * case['deg']
        return dict(bytes=16 * ng * b + v4, flops=_series(ng, b, terms))
    if kind in ('tdh', 'tdh_xi'):
        ns, v = case['samples'], case['samples'] * case['n_eta']
        npts = ng if kind == 'tdh' else case['n_xi']
        return dict(bytes=8 * ng * v + v4 * (ns + 1) + 4 * npts * ns * (case['steps'] + 1),
                    flops=_series(ng, 2 * v, case['steps'] * case['deg']))
    if kind == 'sigma':
        ns = case['samples']
        return dict(bytes=ng * (32 * ns + 8 * ns * (case['steps'] + 1)) + 2 * v4,
                    flops=_series(ng, 2 * ns, case['steps'] * case['deg']))
    if kind == 'time_order':
        m = 4
        while m < 4 * (case['steps'] + 1):
            m *= 2
        p = case['points'] * case['samples']
        return dict(bytes=12 * p * (case['steps'] + 1), flops=p * 7.5 * m * math.log2(m))
    if kind == 'whole':
        ns = case['samples'] * case['group']
        vt = (case['n_eta'] + 1) * case['n_cheb'] + 2 * (case['n_eta'] + 1) * case['steps'] * case['deg']
        return dict(bytes=3 * v4 + ns * 32 * (case['steps'] + 1), flops=_series(ng, ns, vt))
    h, p = case['width'], case['n_in'] * case['width'] + 2 * case['width'] ** 2 + case['width'] * case['n_out']
    return dict(bytes=4 * (case['rows'] * (case['n_in'] + case['n_out']) + case['cheap'] * (case['n_in'] + case['n_out'])
                           + 2 * (p + 3 * h + case['n_out'])), flops=6 * p * case['rows'] + 2 * p * case['cheap'])


def tolerance(case):
    """Relative 2-norm errors, about four times what the 32-bit path shows against `exact` (measured:
    apply_h 2.7e-7, propagate 7e-7, split 1.4e-6, filter 1e-5 at degree 233, tdh 5e-7, tdh_xi 1.5e-6, sigma
    2.4e-6, time_order 1e-7, whole 3e-6; the network's bf16 products 6e-3)."""
    return dict(rel=dict(apply_h=1e-6, propagate=3e-6, split=6e-6, filter=4e-5, tdh=3e-6, tdh_xi=6e-6, sigma=1e-5,
                         time_order=5e-7, whole=1.5e-5, net=2.5e-2)[case['kind']])


# ------------------------------------------------------------------ 64-bit restatement
def _k2(n, h, dtype):
    k = 2 * math.pi * torch.fft.fftfreq(n, d=h, device=DEV, dtype=F64)
    return (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).to(dtype)


class _Exact:
    """H = |k|^2/2 + V + sum_ap beta E dV <beta| and the method's steps, on [n, n, n] complex128."""

    def __init__(self, n):
        s = _system(n)
        self.n, self.h, self.dV = n, s['h'], s['h'] ** 3
        self.k2 = _k2(n, s['h'], F64)
        self.vc = torch.where(self.k2 > 0, 4 * math.pi / torch.clamp(self.k2, min=1e-30), torch.zeros_like(self.k2))
        self.v = torch.as_tensor(s['vloc'].astype(np.float32)).to(DEV).to(F64)
        self.kb = None
        if s['kb_atoms']:
            m, na = max(len(a[0]) for a in s['kb_atoms']), len(s['kb_atoms'])
            idx, beta, e = np.zeros((na, m), np.int64), np.zeros((na, m, 4), np.float32), np.zeros((na, 4), np.float32)
            for a, (sup, b, ee) in enumerate(s['kb_atoms']):
                idx[a, :len(sup)], beta[a, :len(sup), :len(ee)], e[a, :len(ee)] = sup, np.asarray(b).T, ee
            self.kb = tuple(torch.as_tensor(t).to(DEV) for t in (idx, beta, e))
        self.lo, self.hi = _spectrum(n)
        self.mid, self.half = 0.5 * (self.hi + self.lo), 0.5 * (self.hi - self.lo)

    def apply(self, x, dv=None):
        y = torch.fft.ifftn(0.5 * self.k2 * torch.fft.fftn(x)) + (self.v if dv is None else self.v + dv) * x
        if self.kb is not None:
            idx, beta, e = self.kb
            flat, step = torch.view_as_real(x.reshape(-1)), 512
            out = torch.view_as_real(y.reshape(-1))
            for a in range(0, idx.shape[0], step):
                i, b = idx[a:a + step], beta[a:a + step].to(F64)
                c = e[a:a + step, :, None].to(F64) * self.dV * torch.bmm(b.transpose(1, 2), flat[i])
                out.index_add_(0, i.reshape(-1), torch.bmm(b, c).reshape(-1, 2))
        return y

    def ht(self, x, dv=None):
        return (self.apply(x, dv) - self.mid * x) / self.half

    def series(self, x, c):
        a, b = x, self.ht(x)
        acc = c[0] * a + c[1] * b
        for k in range(2, len(c)):
            a, b = b, 2 * self.ht(b) - a
            acc = acc + c[k] * b
        return acc

    def prop_coeffs(self, dt, deg):
        # (2 - delta_k0) (-i)^k J_k(a), J_k(a) = (1/pi) int_0^pi cos(k t - a sin t) dt by the
        # trapezoid rule (exact to rounding for a periodic integrand)
        a, t = self.half * abs(dt), (np.arange(512) + 0.5) * math.pi / 512
        k = np.arange(deg + 1)
        j = np.cos(k[:, None] * t[None, :] - a * np.sin(t)[None, :]).mean(axis=1)
        c = np.where(k == 0, 1.0, 2.0) * (-1j) ** k * j
        c = np.conj(c) if dt < 0 else c
        return [complex(v) for v in c], complex(np.exp(-1j * self.mid * dt))

    def step(self, x, dt, deg):
        c, ph = self.prop_coeffs(dt, deg)
        return ph * self.series(x, c)

    def step_pair(self, x, d, dvh, dv, dt, deg):
        """One step of a vector and of its derivative along the potential dv."""
        c, ph = self.prop_coeffs(dt, deg)
        a, da = x, d
        b, db = self.ht(x, dvh), self.ht(d, dvh) + dv / self.half * x
        s, ds = c[0] * a + c[1] * b, c[0] * da + c[1] * db
        for k in range(2, len(c)):
            nb = 2 * self.ht(b, dvh) - a
            ndb = 2 * self.ht(db, dvh) + 2 * dv / self.half * b - da
            a, b, da, db = b, nb, db, ndb
            s, ds = s + c[k] * b, ds + c[k] * db
        return ph * s, ph * ds

    def poisson(self, f):
        return torch.fft.ifftn(self.vc * torch.fft.fftn(f)).real

    def tdh(self, eta, source, steps, dt, deg):
        """u^R(t_j), [steps + 1, n, n, n], of one sample's real or complex orbitals."""
        n, w = self.n, 2.0 / eta.shape[0]
        e = [x.to(C128).view(n, n, n) for x in eta]
        vp = self.poisson(source.to(F64).view(n, n, n))
        d = [-1j * vp * x for x in e]
        out = []
        for j in range(steps + 1):
            rho = w * sum(x.real ** 2 + x.imag ** 2 for x in e)
            dr = w * sum(2 * (x.conj() * y).real for x, y in zip(e, d))
            if j == 0:
                rho0 = rho
            dvh, dv = self.poisson(rho - rho0), self.poisson(dr)
            out.append(dv)
            if j < steps:
                pairs = [self.step_pair(x, y, dvh, dv, dt, deg) for x, y in zip(e, d)]
                e, d = [p[0] for p in pairs], [p[1] for p in pairs]
        return torch.stack(out)

    def sigma(self, zocc, zun, u, phi, steps, dt, deg):
        n = self.n
        zp, zm, f = zun.to(C128).view(n, n, n), zocc.to(C128).view(n, n, n), phi.to(F64).view(n, n, n)
        out = torch.zeros(2 * steps + 1, dtype=C128, device=DEV)
        for j in range(steps + 1):
            uj = u[j].to(C128).view(n, n, n)
            sp, sm = self.dV * (f * zp * uj).sum(), -self.dV * (f * zm * uj).sum()
            if j == 0:
                out[steps] = 0.5 * (sp + sm)
            else:
                out[steps + j], out[steps - j] = sp, sm
            if j < steps:
                zp, zm = self.step(zp, dt, deg), self.step(zm, -dt, deg)
        return out, torch.stack([zm.reshape(-1), zp.reshape(-1)])

    def split(self, x, steps, dt):
        """The symmetric split-operator step, KB factors atom by atom in greedy colours."""
        fac = []
        if self.kb is not None:
            idx, beta, e = self.kb
            used, col = {}, []
            sup = [set(int(i) for i in atom[0]) for atom in _system(self.n)['kb_atoms']]
            for a, pts in enumerate(sup):
                taken = {c for c, grid in used.items() if grid & pts}
                c = next(k for k in range(64) if k not in taken)
                used.setdefault(c, set()).update(pts)
                col.append(c)
            order = sorted(range(len(col)), key=lambda a: (col[a], a))
            for a in order:
                r = math.sqrt(self.dV) * beta[a].to(F64)
                p = int((beta[a].abs().sum(0) > 0).sum())
                q, m = torch.linalg.qr(r[:, :p])
                mm = m @ torch.diag(e[a, :p].to(F64)) @ m.T
                w, vec = torch.linalg.eigh(mm)
                f = vec.to(C128) @ torch.diag(torch.exp(-0.5j * dt * w) - 1) @ vec.T.to(C128)
                fac.append((idx[a], q.to(C128), f))
        half = torch.exp(-0.5j * dt * self.v)
        kin = torch.exp(-0.5j * dt * self.k2)

        def kb(y, fs):
            flat = y.reshape(-1).clone()
            for i, q, f in fs:
                d = q @ (f @ (q.T @ flat[i]))
                flat.index_add_(0, i, d)
            return flat.view(y.shape)
        for _ in range(steps):
            x = kb(x, fac)
            x = half * torch.fft.ifftn(kin * torch.fft.fftn(half * x))
            x = kb(x, fac[::-1])
        return x


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 words of int64 tensors holding 32-bit counters."""
    M = 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M) ^ c1 ^ k0, p1 & M, ((p0 >> 32) & M) ^ c3 ^ k1, p0 & M
    return c0, c1, c2, c3


def _philox_noise(n, h, seed, stream, sample, vec):
    blk = torch.arange((n ** 3 + 3) // 4, device=DEV, dtype=torch.int64)
    one = torch.ones_like(blk)
    w = torch.stack(_philox(blk, one * vec, one * sample, one * stream, seed & 0xFFFFFFFF, seed >> 32), dim=1)
    return (1 - 2 * (w.reshape(-1)[:n ** 3] >> 31)).to(F64) * h ** -1.5


def _time_order(uR):
    """Time ordering along axis 0 in 64 bits."""
    nt, m = uR.shape[0], 4
    while m < 4 * nt:
        m *= 2
    out = torch.empty(uR.shape, dtype=C128, device=DEV)
    for p in range(0, uR.shape[1], 32768):
        x = torch.zeros(m, min(32768, uR.shape[1] - p), dtype=C128, device=DEV)
        x[:nt] = uR[:, p:p + 32768]
        X = torch.fft.ifft(x, dim=0) * m
        X[m // 2 + 1:] = X[m // 2 + 1:].conj().clone()
        out[:, p:p + 32768] = torch.fft.fft(X, dim=0)[:nt] / m
    return out


def _xi_project(ex, f, case, sample):
    seed, stream, _, n_xi, f_g, L = _xi(case)
    ng = case['n'] ** 3
    K = max(1, int(math.floor(ng * f_g / L + 0.5)))
    c = 1.0 / math.sqrt(n_xi * K * L * ex.dV / ng)
    k = torch.arange(K, device=DEV, dtype=torch.int64)
    lane = torch.arange(L, device=DEV, dtype=torch.int64)
    out = torch.empty(f.shape[0], n_xi, dtype=F64, device=DEV)
    step = max(1, 10 ** 7 // (K * L))
    for m0 in range(0, n_xi, step):
        m = torch.arange(m0, min(n_xi, m0 + step), device=DEV, dtype=torch.int64)
        kk = k[None, :].expand(len(m), K)
        one = torch.ones_like(kk)
        w0, w1, _, _ = _philox(kk, m[:, None].expand(len(m), K), one * sample, one * stream, seed, 0)
        r = ((w0 * (ng // L)) >> 32)[:, :, None] * L + lane
        s = (1 - 2 * ((w1[:, :, None] >> lane) & 1)).to(F64)
        for j in range(f.shape[0]):
            out[j, m0:m0 + len(m)] = c * ex.dV * (s * f[j].reshape(-1)[r]).sum((1, 2))
    return out


def _exact_net(case, st):
    dims = [case['n_in']] + 3 * [case['width']] + [case['n_out']]
    p, off, ws = torch.as_tensor(st['params']).to(DEV).to(F64), 0, []
    for a, b in zip(dims[:-1], dims[1:]):
        ws.append((p[off:off + a * b].view(a, b), p[off + a * b:off + a * b + b]))
        off += a * b + b

    def forward(x):
        acts = [x.to(F64)]
        for i, (w, b) in enumerate(ws):
            z = acts[-1] @ w + b
            acts.append(torch.tanh(z) if i < 3 else z)
        return acts
    acts = forward(st['x'])
    e = acts[-1] - st['t'].to(F64)
    d, grads = 2 * e / e.numel(), []
    for i in range(3, -1, -1):
        grads = [(acts[i].T @ d).reshape(-1), d.sum(0)] + grads
        if i:
            d = (d @ ws[i][0].T) * (1 - acts[i] ** 2)
    return dict(loss=float((e * e).mean()), grads=torch.cat(grads), y=forward(st['xc'])[-1])


def _exact_qp(case, sig, xs):
    n, dt, eps, window, step = case['steps'], 0.05, -0.15, 2.0, 1e-3
    t = dt * np.arange(-n, n + 1)
    w = np.ones(2 * n + 1)
    w[0] = w[-1] = 0.5
    damped = dt * w * sig.mean(0).cpu().numpy() * np.exp(-0.5 * (3.0 / (n * dt)) ** 2 * t ** 2)
    xm = float(xs.mean())
    f = lambda e: e - eps - xm - float((np.exp(1j * e * t) * damped).sum().real)
    om = eps - window + step * np.arange(int(round(2 * window / step)) + 1)
    v = om - eps - xm - (np.exp(1j * np.outer(om, t)) @ damped).real
    i = np.nonzero(np.sign(v[:-1]) * np.sign(v[1:]) <= 0)[0]
    if len(i) == 0:
        return None
    i = i[np.argmin(np.abs(0.5 * (om[i] + om[i + 1]) - eps))]
    a, b, fa = om[i], om[i + 1], v[i]
    while b - a > 1e-10:
        c = 0.5 * (a + b)
        fc = f(c)
        if np.sign(fc) == np.sign(fa) and fc != 0:
            a, fa = c, fc
        else:
            b = c
    return 0.5 * (a + b)


def exact(case, seed):
    kind, st = case['kind'], _inputs(case, seed)
    if kind == 'time_order':
        return torch.stack([_time_order(r.to(F64)) for r in st['uR']])
    if kind == 'net':
        return _exact_net(case, st)
    n = case['n']
    if kind == 'filter' and n ** 3 * case['batch'] * case['n_cheb'] > 4 * 10 ** 9:
        return None
    ex = _Exact(n)
    if kind in ('apply_h', 'filter', 'propagate', 'split'):
        out = torch.empty(st['x'].shape, dtype=C128, device=DEV)
        dirs = _dirs(case['batch'])
        for b in range(case['batch']):
            x = st['x'][b].to(C128).view(n, n, n)
            if kind == 'apply_h':
                x = ex.apply(x)
            elif kind == 'filter':
                x = ex.series(x, [float(a) for a in _filter_coeffs(case)])
            elif kind == 'split':
                if n == 128:             # 657 atoms one after another: too slow here
                    return None
                x = ex.split(x, case['steps'], 0.05 * int(dirs[b]))
            else:
                for _ in range(case['steps']):
                    x = ex.step(x, 0.05 * int(dirs[b]), case['deg'])
            out[b] = x.reshape(-1)
        return out
    if kind in ('tdh', 'tdh_xi'):
        rows = []
        for s in range(case['samples']):
            u = ex.tdh(st['eta'][s * case['n_eta']:(s + 1) * case['n_eta']], st['source'][s], case['steps'], 0.05,
                       case['deg'])
            rows.append(u.reshape(case['steps'] + 1, -1) if kind == 'tdh' else _xi_project(ex, u, case, s))
        return torch.stack(rows)
    if kind == 'sigma':
        r = [ex.sigma(st['z'][2 * s], st['z'][2 * s + 1], st['u'][s], st['phi'], case['steps'], 0.05, case['deg'])
             for s in range(case['samples'])]
        return dict(sigma=torch.stack([a for a, _ in r]), zeta=torch.cat([z for _, z in r]))
    phi, co, ne = _phi(n), [float(a) for a in _filter_coeffs(case)], case['n_eta']
    sig, xs = [], []
    for s in range(case['samples'] * case['group']):
        z = [_philox_noise(n, ex.h, int(seed) + 1, 1, s, v) for v in range(ne + 1)]
        p = [ex.series(v.to(C128).view(n, n, n), co).reshape(-1) for v in z]
        uR = ex.tdh(torch.stack(p[1:]), z[0] * phi, case['steps'], 0.05, case['deg'])
        u = _time_order(uR.reshape(case['steps'] + 1, -1))
        sig.append(ex.sigma(p[0], z[0] - p[0], u, phi, case['steps'], 0.05, case['deg'])[0])
        f = [torch.fft.fftn((phi * v).view(n, n, n)) for v in p[1:]]
        xs.append(-sum((ex.vc * (a.real ** 2 + a.imag ** 2)).sum() for a in f) * ex.dV / n ** 3 / ne)
    sig, xs = torch.stack(sig), torch.stack(xs)
    return dict(sigma=sig, x=xs, eps_qp=_exact_qp(case, sig, xs))
