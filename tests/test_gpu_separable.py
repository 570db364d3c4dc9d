"""The separable kinetic path (contexts without a cutoff) against the transform path: a cutoff above
every kinetic energy selects the latter and changes no operator, so the two agree to rounding on every
grid, batch and KB form; and planes with more KB slots or colours than the separable step has room for."""
import numpy as np
import pytest

from oracle import chebyshev as cheb
from oracle import hamiltonian as ham
from oracle import splitop
from paper_2601_21005_gb300 import build, synth

import gpu_common as gc

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


def _ctx(s, batch, ecut, kb):
    from paper_2601_21005_gb300 import sgw
    c = sgw.Context(s['n'], s['h'], ecut=ecut, max_batch=batch)
    c.set_potential(gc.to_dev(s['vloc'].ravel(), torch, torch.float32), s['kb_atoms'] if kb else [])
    c.set_spectrum(float(s['vloc'].min()) - 2.0, 0.5 * 3 * (np.pi / s['h']) ** 2 + 2.0)
    return c


def _system(n):
    if n == 16:
        s = synth.wells(n=16, h=0.6)
        # two atoms of one and two projectors whose spheres overlap and wrap around the box
        s['kb_atoms'] = [synth.kb_projectors(16, 0.6, (0.5, 9.0, 4.8), 0.9, (1.2,), 0),
                         synth.kb_projectors(16, 0.6, (1.7, 8.1, 4.2), 0.8, (0.7, -0.3), 1)]
        return s
    hp = dict(synth.H_PARAMS)
    hp['Es'] = 0.3
    return synth.si_cluster(n=n, h=0.5, radius=4.5, hp=hp)


# Rounding of one H application relative to its largest element: a chain of at most 6 line transforms
# of depth log2 n <= 9 and a few sums, each adding at most 2^-24 of a value below |T|max |b|; their
# random sum stays below 4 sqrt(6 * 9) 2^-24 = 1.8e-6 of it.  Sixteen terms of a propagation step
# add at most in proportion.
TOL_H = 1.8e-6


@pytest.mark.parametrize('n', [16, 32, 48, 64, 96, 128, 288])
@pytest.mark.parametrize('kb', [True, False])
def test_separable_matches_the_transform_path(n, kb):
    assert torch.cuda.is_available()
    build.build()
    s = _system(n)
    B = 3 if n < 288 else 2
    g = torch.Generator(device='cuda').manual_seed(n)
    x = torch.randn(B, n ** 3, dtype=torch.complex64, device='cuda', generator=g)
    outs = []
    for ecut in (0.0, 1e6):
        c = _ctx(s, 4, ecut, kb)
        y = torch.empty_like(x)
        c.apply_h(x, y)
        p = x.clone()
        c.propagate(p, 2, 0.05, 16, np.array([1, -1, 1], dtype=np.int8)[:B])
        f = torch.empty_like(x)
        c.filter_occupied(np.array([0.3, -0.2, 0.1]), x, f)          # the shortest plans: degrees 2 and 1
        f1 = torch.empty_like(x)
        c.filter_occupied(np.array([0.3, -0.2]), x, f1)
        uR = torch.empty(1, 3, n ** 3, dtype=torch.float32, device='cuda')
        src = x[0].real.contiguous()
        c.tdh_response((0.05 * x[:2]).contiguous(), src, 1, 2, 2, 0.05, 10, uR)
        torch.cuda.synchronize()
        outs.append((y, p, f, f1, uR))
        c.close()
    for a, b, terms in zip(outs[0], outs[1], (1, 32, 2, 1, 40)):
        assert float((a - b).abs().max() / b.abs().max()) < TOL_H * terms


@pytest.mark.parametrize('n', [16, 32, 48, 64, 96])
def test_cutoff_that_binds(n):
    """A cutoff below the largest kinetic energy of one axis caps T(k), which is then no sum over the axes:
    H psi, a propagation step and a split-operator step against the oracle with the same cap.  (Rounding of
    H psi as above; a step's as in the parity tests.)"""
    build.build()
    s = _system(n)
    ecut = 0.3 * 0.5 * (np.pi / s['h']) ** 2
    g, kb = ham.Grid(n, s['h'], ecut), ham.KB(s['kb_atoms'])
    lo, hi = float(s['vloc'].min()) - 2.0, ecut + 4.0
    r = np.random.default_rng(n)
    x = (r.normal(size=(2,) + g.shape()) + 1j * r.normal(size=(2,) + g.shape())).astype(np.complex64)
    c = _ctx(s, 2, ecut, True)
    c.set_spectrum(lo, hi)
    xd = gc.to_dev(x.reshape(2, -1), torch, torch.complex64)
    y, p = torch.empty_like(xd), xd.clone()
    c.apply_h(xd, y)
    c.propagate(p, 1, 0.05, 12, np.array([1, -1], dtype=np.int8))
    h = lambda v: ham.apply_h(v, g, s['vloc'], kb)
    assert gc.rel_err(y.cpu().numpy().reshape(x.shape), h(x.astype(np.complex128))) < TOL_H
    for b, d in enumerate((1, -1)):
        ref = cheb.propagate_step(h, x[b].astype(np.complex128), lo, hi, 0.05 * d, 12)
        assert gc.rel_err(p[b].cpu().numpy().reshape(g.shape()), ref) < 1e-5
    if n in (16, 32, 64):
        q = xd.clone()
        c.propagate_split(q, 1, 0.05)
        ref = splitop.split_propagate(x[0].astype(np.complex128), g, s['vloc'], splitop.KBSplit(s['kb_atoms'], g), 0.05, 1)
        assert gc.rel_err(q[0].cpu().numpy().reshape(g.shape()), ref) < 1e-5


def test_more_slots_than_the_separable_step_holds():
    """3090 one-point atoms in one 128^2 plane: above the separable step's 3072 slots, within the
    transform path's 3104, so the context falls back to it.  V_NL is then diagonal."""
    from paper_2601_21005_gb300 import sgw
    build.build()
    n, h, na, e, beta = 128, 0.5, 3090, 0.4, 1.3
    pts = 5 * np.arange(na)                                  # z = 0
    atoms = [(np.array([p]), np.full((1, 1), beta), np.array([e])) for p in pts]
    g = torch.Generator(device='cuda').manual_seed(1)
    v = torch.randn(n ** 3, device='cuda', generator=g)
    x = torch.randn(2, n ** 3, dtype=torch.complex64, device='cuda', generator=g)
    a = sgw.Context(n, h, max_batch=2)
    a.set_potential(v, atoms)
    ya = torch.empty_like(x)
    a.apply_h(x, ya)
    w = v.clone()
    w[torch.as_tensor(pts, device='cuda')] += e * beta * beta * h ** 3
    b = sgw.Context(n, h, max_batch=2)
    b.set_potential(w)
    yb = torch.empty_like(x)
    b.apply_h(x, yb)
    assert float((ya - yb).abs().max() / yb.abs().max()) < TOL_H
    a.set_potential(w)                                       # without the atoms the separable step is back
    a.apply_h(x, ya)
    assert torch.equal(ya, yb)


def _colours(atoms, unit, ng):
    """Most colours that first-fit colouring of the atoms takes in a unit of `unit` points."""
    most = 0
    for u in range(ng // unit):
        used = {}
        for idx, _, _ in atoms:
            pts = idx[(idx >= u * unit) & (idx < (u + 1) * unit)]
            taken = set().union(*[used.get(p, set()) for p in pts]) if len(pts) else set()
            c = next(i for i in range(len(atoms)) if i not in taken)
            for p in pts:
                used.setdefault(p, set()).add(c)
            most = max(most, c + 1) if len(pts) else most
    return most


def test_more_colours_than_the_separable_step_holds():
    """33 pairs of atoms a_i, b_i where a_i and b_j share a point of one 48^2 plane for all i != j: first-fit
    colouring in the order a_0 b_0 a_1 ... takes 33 colours in the plane, but few in units of 8 rows, which
    the transform path has.  (a_0 and b_0 share a point elsewhere, so the atoms as a whole take 2.)"""
    from paper_2601_21005_gb300 import sgw
    build.build()
    n, h, m = 48, 0.5, 33
    r = np.random.default_rng(3)
    pairs = [(i, j) for i in range(m) for j in range(m) if i != j]
    pts = {p: int(q) for p, q in zip(pairs, r.permutation(n * n))}
    atoms = []
    for i in range(m):
        for own in ([pts[i, j] for j in range(m) if j != i], [pts[j, i] for j in range(m) if j != i]):
            idx = np.sort(np.array(own + ([n * n] if i == 0 else [])))
            atoms.append((idx, r.uniform(0.3, 1.0, (1, len(idx))), np.array([r.uniform(-1, 1)])))
    assert _colours(atoms, n * n, 2 * n * n) == 33 and _colours(atoms, 8 * n, 2 * n * n) <= 32
    assert _colours(atoms, 2 * n * n, 2 * n * n) == 2
    v = r.normal(size=(n, n, n)).astype(np.float32)
    x = (r.normal(size=(2, n, n, n)) + 1j * r.normal(size=(2, n, n, n))).astype(np.complex64)
    c = sgw.Context(n, h, max_batch=2)
    c.set_potential(gc.to_dev(v.ravel(), torch, torch.float32), atoms)
    xd = gc.to_dev(x.reshape(2, -1), torch, torch.complex64)
    y = torch.empty_like(xd)
    c.apply_h(xd, y)
    ref = ham.apply_h(x.astype(np.complex128), ham.Grid(n, h), v.astype(np.float64), ham.KB(atoms))
    assert gc.rel_err(y.cpu().numpy().reshape(ref.shape), ref) < TOL_H
    # 33 atoms at one point are refused on every path
    with pytest.raises(RuntimeError):
        c.set_potential(gc.to_dev(v.ravel(), torch, torch.float32), [(np.array([5]), np.ones((1, 1)), np.ones(1))] * 33)


@pytest.mark.parametrize('n', [16, 32, 64, 128])
def test_split_steps_match_the_transform_path(n):
    """Propagation, TDH and Sigma(t) by split-operator steps with and without a (never reached) cutoff, and
    one call of three steps against three calls of one (merged colours against halves)."""
    build.build()
    s = _system(n)
    B = 3
    g = torch.Generator(device='cuda').manual_seed(n)
    x = torch.randn(B, n ** 3, dtype=torch.complex64, device='cuda', generator=g)
    outs = []
    for ecut in (0.0, 1e6):
        c = _ctx(s, 4, ecut, True)
        dirs = np.array([1, -1, 1], dtype=np.int8)
        p, q = x.clone(), x.clone()
        c.propagate_split(p, 3, 0.05, dirs)
        for _ in range(3):
            c.propagate_split(q, 1, 0.05, dirs)
        uR = torch.empty(1, 3, n ** 3, dtype=torch.float32, device='cuda')
        c.tdh_response((0.05 * x[:2]).contiguous(), x[0].real.contiguous(), 1, 2, 2, 0.05, 0, uR)
        z = x[:2].clone()
        sig = torch.empty(1, 5, dtype=torch.complex128, device='cuda')
        c.sigma_c(z, x[2].real.contiguous(), x[:3].reshape(1, 3, -1).contiguous(), 1, 2, 0.05, 0, sig)
        torch.cuda.synchronize()
        assert float((p - q).abs().max() / q.abs().max()) < 3 * 4 * TOL_H
        outs.append((p, uR, z))
        c.close()
    # a step is 6 line transforms and the phases, twice the chain of one H application
    for a, b, steps in zip(outs[0], outs[1], (3, 6, 2)):
        assert float((a - b).abs().max() / b.abs().max()) < 4 * TOL_H * steps
