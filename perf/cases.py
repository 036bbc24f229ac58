"""Workloads of the library, as programs use it, and their values in 64 bits.

A case is one call (or one pass of a simulation loop) through the public binding:

  mobility    [U; E] = M [F; S], cube or sheared cell, mixed or FP64
  mobility11  [U; Omega; E] = M [F; L; S] (handles with torque = 1)
  sample      Brownian slip velocities, in-kernel noise
  step        one constrained mid-point step, with or without the overlap force
  rfd         one Euler-Maruyama step with the random-finite-difference drift
  batch       one step of many independent suspensions in one handle
  serve       a burst of mobility / sample / step requests to the serving loop, host arrays

a = eta = kT = 1 throughout; a step starts from the same x_k on every pass.
`exact` restates the method in FP64 with torch alone (same cutoffs, grids,
stopping rules and noise streams; see the definitions in include/pse.h).
"""
import math
import random

import numpy as np
import torch

import paper_1709_06946_gb300 as pse

DT = 1e-3
SPRING = 1000.0   # overlap force constant k (kT / a^2)


# ------------------------------------------------------------------ the cases
def _case(name, call, n, phi, **kw):
    c = {'name': name, 'call': call, 'n': n, 'phi': phi, 'tol': 1e-3, 'xi': 0.5, 'precision': 'mixed', 'strain': 0.0,
         'graph': False, 'overlap': 0.0, 'nsys': 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest suspensions: a single product of a resolved-hydrodynamics code, launch and latency bound
        _case('mobility_1k', 'mobility', 1000, 0.1),
        # the all-FP64 form, used to validate a mixed-precision run; odd particle count
        _case('mobility_11k_fp64', 'mobility', 11003, 0.25, precision='fp64'),
        # Lees-Edwards shear at strain 1/2: lattice weights, support P = 10
        _case('mobility_sheared_150k', 'mobility', 150001, 0.3, strain=0.5),
        # the grand mobility of the largest suspension the benchmark names
        _case('mobility_1m', 'mobility', 1048576, 0.3),
        # forces, torques and stresslets: the 11-moment product
        _case('mobility11_100k', 'mobility11', 100000, 0.2),
        # Brownian velocities at the tighter tolerance of the serving stream (P = 8, more Lanczos steps)
        _case('sample_50k_tight', 'sample', 50000, 0.25, tol=1e-4),
        # a production loop with hard-sphere repulsion: overlap force, then the graph-captured step
        _case('step_3k_force', 'step', 3000, 0.3, graph=True, overlap=0.05),
        # the static-structure runs of the equilibrium validation: ideal spheres, overlaps allowed
        _case('step_64k_ideal', 'step', 64000, 0.5, xi=0.6, graph=True),
        # the headline workload: one graph-captured step of 2^20 spheres
        _case('step_1m', 'step', 1048576, 0.3, graph=True),
        # the alternative integrator: three stresslet solves and two extra neighbour lists per step
        _case('rfd_30k', 'rfd', 30011, 0.2),
        # many small suspensions advanced in lockstep by one handle
        _case('batch_64', 'batch', 2500, 0.2, nsys=64),
        # six concurrent requests over host arrays, two of each kind, on resident suspensions
        _case('serve_burst', 'serve', 6000, 0.25, nsys=6),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    call = rng.choice(['mobility', 'mobility', 'sheared', 'fp64', 'mobility11', 'sample', 'sample', 'step', 'step',
                       'step', 'rfd', 'batch', 'serve'])
    phi = round(rng.uniform(0.08, 0.3), 3)
    tol = rng.choice([1e-3, 1e-3, 1e-4])
    if call == 'mobility':
        c = _case('', 'mobility', size(1000, 1000000), phi, tol=tol, xi=round(rng.uniform(0.45, 0.6), 3))
    elif call == 'sheared':
        c = _case('', 'mobility', size(3000, 300000), phi, strain=round(rng.uniform(0.1, 0.5), 2))
    elif call == 'fp64':
        c = _case('', 'mobility', size(1000, 30000), phi, tol=tol, precision='fp64')
    elif call == 'mobility11':
        c = _case('', 'mobility11', size(1000, 250000), phi)
    elif call == 'sample':
        c = _case('', 'sample', size(1000, 250000), phi, tol=tol)
    elif call == 'step':
        c = _case('', 'step', size(1000, 500000), phi, tol=rng.choice([1e-3, 1e-3, 1e-3, 1e-4]),
                  graph=rng.random() < 0.7, overlap=rng.choice([0.0, 0.05]))
    elif call == 'rfd':
        c = _case('', 'rfd', size(1000, 60000), phi)
    elif call == 'batch':
        c = _case('', 'batch', size(1200, 6000), phi, nsys=rng.randrange(8, 97))
    else:
        c = _case('', 'serve', size(2000, 20000), phi, nsys=6)
    del c['name']
    return c


def _sizes(case):
    """Particle counts and volume fractions of a case's suspensions (spread over a factor of 8 around n)."""
    k = case['nsys']
    if k == 1:
        return [(case['n'], case['phi'])]
    r = random.Random(1000 * k + case['n'])
    return [(int(case['n'] * 8.0 ** r.uniform(-0.5, 0.5)), min(0.3, case['phi'] * r.uniform(0.5, 1.5))) for _ in range(k)]


def _deform(case):
    return None if not case['strain'] else np.array([[1.0, case['strain'], 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])


# ------------------------------------------------------------------ inputs
def _box(n, phi):
    return (4.0 * math.pi * n / (3.0 * phi)) ** (1.0 / 3.0)


def _spheres(n, L, seed):
    """Hard-sphere centres (n x 3, FP64) by random sequential addition in rounds on the GPU: cells that
    hold at most one centre, a proposal is dropped when it touches a placed sphere or an earlier proposal."""
    g = torch.Generator(device='cuda').manual_seed(seed)
    nc = math.ceil(L * math.sqrt(3.0) / 2.0)
    held = torch.full((nc ** 3,), -1, dtype=torch.int64, device='cuda')      # placed sphere of a cell
    pos = torch.empty((n, 3), dtype=torch.float64, device='cuda')
    o = torch.arange(-2, 3, device='cuda')
    off = torch.stack(torch.meshgrid(o, o, o, indexing='ij'), -1).reshape(-1, 3)
    off = off[(off != 0).any(1)]
    m = max(256, min(1 << 18, n))
    none = torch.iinfo(torch.int64).max
    placed = 0
    while placed < n:
        x = torch.rand((m, 3), generator=g, dtype=torch.float64, device='cuda') * L
        c = (x * (nc / L)).long().clamp_(max=nc - 1)
        flat = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
        free = (held[flat] < 0).nonzero()[:, 0]
        first = torch.full((nc ** 3,), none, dtype=torch.int64, device='cuda')
        first.scatter_reduce_(0, flat[free], free, 'amin')
        k = free[first[flat[free]] == free]
        q = (c[k][:, None, :] + off) % nc
        q = (q[..., 0] * nc + q[..., 1]) * nc + q[..., 2]
        ok = torch.ones(len(k), dtype=torch.bool, device='cuda')
        for who, at in ((held[q], pos), (first[q], x)):
            near = (who >= 0) & (who != none)
            if at is x:
                near &= who < k[:, None]
            d = x[k][:, None, :] - at[torch.where(near, who, 0)]
            d -= L * torch.round(d / L)
            ok &= ~(near & ((d * d).sum(-1) < 4.0)).any(1)
        k = k[ok][:n - placed]
        pos[placed:placed + len(k)] = x[k]
        held[flat[k]] = torch.arange(placed, placed + len(k), device='cuda')
        placed += len(k)
    return pos


def _positions(case, n, phi, L, seed):
    g = torch.Generator(device='cuda').manual_seed(seed + 7)
    if phi > 0.31:   # ideal spheres: uniform, overlaps allowed
        return torch.rand((n, 3), generator=g, dtype=torch.float64, device='cuda') * L
    x = _spheres(n, L, seed)
    if case['overlap']:   # as a run with a soft repulsion leaves them: small overlaps
        x = (x + case['overlap'] * torch.randn((n, 3), generator=g, dtype=torch.float64, device='cuda')) % L
    A = _deform(case)
    return x if A is None else x @ torch.tensor(A.T.copy(), device='cuda')


def _inputs(case, seed):
    """Per suspension: N, L, positions (FP64) and moments F, Lt, S in the handle's precision."""
    dt = torch.float64 if case['precision'] == 'fp64' else torch.float32
    out = []
    for q, (n, phi) in enumerate(_sizes(case)):
        s = (seed * 100003 + 977 * q + 1) % (1 << 31)
        L = _box(n, phi)
        g = torch.Generator(device='cuda').manual_seed(s + 3)
        F, Lt, S = (torch.randn((n, w), generator=g, dtype=torch.float64, device='cuda').to(dt) for w in (3, 3, 5))
        out.append({'n': n, 'L': L, 'pos': _positions(case, n, phi, L, s), 'F': F, 'Lt': Lt, 'S': S})
    return out


def prepare(case, seed):
    ins = _inputs(case, seed)
    st = {'case': case, 'seed': seed, 'ins': ins}
    opts = {'xi': case['xi'], 'tol': case['tol'], 'precision': case['precision']}
    if case['call'] == 'serve':
        st['opts'] = opts
        st['srv'] = pse.Server(slots=4, budget_bytes=64 << 30)
        for i in ins:
            for k in ('pos', 'F', 'S'):
                i[k] = i[k].cpu().numpy()
            t, _ = st['srv'].submit('mobility', i['pos'], i['L'], F=i['F'], S=i['S'], **opts)   # makes it resident
            st['srv'].wait(t)
        return st
    if case['strain']:
        opts['deform'] = _deform(case)
    if case['graph']:
        opts['use_graph'] = 1
    if case['call'] == 'mobility11':
        opts['torque'] = 1
    if case['call'] == 'batch':
        st['pos'] = torch.cat([i['pos'] for i in ins])
        st['h'] = pse.PSE([i['n'] for i in ins], [i['L'] for i in ins], **opts)
    else:
        st['h'] = pse.PSE(ins[0]['n'], ins[0]['L'], **opts)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, seed, i = st['case'], st['seed'], st['ins'][0]
    call = case['call']
    if call == 'serve':
        return _serve(st)
    h = st['h']
    if call == 'mobility':
        return h.mobility(i['pos'], i['F'], i['S'])
    if call == 'mobility11':
        return h.mobility11(i['pos'], i['F'], i['Lt'], i['S'])
    if call == 'sample':
        U, E, _ = h.brownian(i['pos'], DT, seed=seed, counter=1)
        return U, E
    if call == 'batch':
        x = st['pos'].clone()
        S, _ = h.step(x, DT, seed=seed, step=1, want_S=True)
        return x, S
    x = i['pos'].clone()
    if call == 'rfd':
        S, _ = h.rfd_step(x, DT, seed=seed, step=1, want_S=True)
        return x, S
    F = h.overlap_force(x, SPRING) if case['overlap'] else None
    S, _ = h.step(x, DT, FP=F, seed=seed, step=1, want_S=True)
    return (x, S) if F is None else (x, S, F)


_KINDS = ('mobility', 'sample', 'step')


def _serve(st):
    srv, seed, opts = st['srv'], st['seed'], st['opts']
    tickets, outs = [], []
    for q, i in enumerate(st['ins']):
        kind = _KINDS[q % 3]
        if kind == 'mobility':
            t, o = srv.submit(kind, i['pos'], i['L'], F=i['F'], S=i['S'], **opts)
        elif kind == 'sample':
            t, o = srv.submit(kind, i['pos'], i['L'], dt=DT, seed=seed, counter=q, **opts)
        else:
            x = i['pos'].copy()
            t, o = srv.submit(kind, x, i['L'], dt=DT, seed=seed, counter=q, **opts)
            o['U'] = x
        tickets.append(t)
        outs.append(o)
    for t in tickets:
        srv.wait(t)
    return [(o['U'], o['S'] if 'S' in o else o['E']) for o in outs]


# ------------------------------------------------------------------ least work
def work(case):
    """Caller's arrays read and written once, and the operations of the method's own counts: per ordered
    pair 178 (full), 130 (S -> E), 68 (S -> U), 260 (11 moments); 2 per support point and component each way;
    2.5 n log2 n per real transform; about 100 per wave vector."""
    ts = 8 if case['precision'] == 'fp64' else 4
    tight = case['tol'] < 5e-4
    nlz, ngm = (10, 9) if tight else (7, 7)
    byts = flops = 0.0
    for q, (n, phi) in enumerate(_sizes(case)):
        p = _Rules(n, _box(n, phi), case['xi'], case['tol'], _deform(case))
        pairs = n * 4.0 / 3.0 * math.pi * p.rcut ** 3 * n / (p.L ** 3)
        n3 = float(p.Ng) ** 3

        def wave(cin, cout):
            return 2.0 * n * p.P ** 3 * (cin + cout) + 2.5 * n3 * math.log2(n3) * (cin + cout) + 50.0 * n3
        full, se, su = 178 * pairs + wave(8, 8), 130 * pairs + wave(5, 5), 68 * pairs + wave(5, 3)
        sample = nlz * 178 * pairs + wave(0, 8)
        call = _KINDS[q % 3] if case['call'] == 'serve' else case['call']
        if call == 'mobility':
            byts += n * (24 + 16 * ts)
            flops += full
        elif call == 'mobility11':
            byts += n * (24 + 22 * ts)
            flops += 260 * pairs + wave(11, 11)
        elif call == 'sample':
            byts += n * (24 + 8 * ts)
            flops += sample
        elif call == 'rfd':
            byts += n * (48 + 5 * ts)
            flops += sample + 3 * ngm * se + 2 * full + 3 * su
        else:
            byts += n * (48 + 5 * ts + (6 * ts if case['overlap'] else 0))
            flops += sample + ngm * se + su + (full if case['overlap'] else 0.0)
    return {'bytes': byts, 'flops': flops}


# ------------------------------------------------------------------ the method in 64 bits
class _Rules:
    """Cutoff, support and grid of a suspension (strict rule, 2^i 3^j grids)."""

    def __init__(self, n, L, xi, tol, A=None):
        self.n, self.L, self.xi, self.tol = n, L, xi, tol
        self.A = np.eye(3) if A is None else A
        G = self.A.T @ self.A
        lam = np.linalg.eigvalsh(G)
        self.lam_min = float(lam[0]) if A is not None else 1.0
        lam_max = float(lam[2]) if A is not None else 1.0
        self.rcut = 1.0 + math.sqrt(math.log(10.0 / tol)) / xi
        lo, hi = 0.0, 800.0   # (1 + u) e^-u = tol
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if (1.0 + mid) * math.exp(-mid) > tol else (lo, mid)
        kcut = 2.0 * xi * math.sqrt(hi)
        P = 1
        while math.exp(-math.pi * P / (2.0 * lam_max)) + math.erfc(math.sqrt(math.pi * P / (2.0 * lam_max))) > tol / 10:
            P += 1
        self.P = P

        def smooth(k, fs):
            for f in fs:
                while k % f == 0:
                    k //= f
            return k == 1

        def up(k, fs):
            while k % 2 or not smooth(k, fs):
                k += 1
            return k
        Ng = up(max(2, math.ceil(kcut * L * math.sqrt(float(G.diagonal().max())) / math.pi - 1e-9)), (2, 3, 5, 7))
        while self._eta(Ng) >= 1.0:
            Ng = up(Ng + 1, (2, 3, 5, 7))
        self.Ng = up(Ng, (2, 3))
        self.h, self.eta = L / self.Ng, self._eta(self.Ng)
        self.V = L ** 3 * float(np.linalg.det(self.A))

    def _eta(self, Ng):
        return (self.L / Ng * self.P * self.xi) ** 2 / (math.pi * self.P)


_I2, _I6 = 1.0 / math.sqrt(2.0), 1.0 / math.sqrt(6.0)


def _sym_y(p, q):
    """Y components of p q^T + q p^T (tuples of x, y, z)."""
    xx, yy, zz = 2 * p[0] * q[0], 2 * p[1] * q[1], 2 * p[2] * q[2]
    r2 = math.sqrt(2.0)
    return [(xx - yy) * _I2, (xx + yy - 2 * zz) * _I6, r2 * (p[0] * q[1] + p[1] * q[0]),
            r2 * (p[0] * q[2] + p[2] * q[0]), r2 * (p[1] * q[2] + p[2] * q[1])]


def _s_mul(s, p):
    """S p for S = sum_k s_k Y_k."""
    xx, yy, zz = s[0] * _I2 + s[1] * _I6, -s[0] * _I2 + s[1] * _I6, -2 * s[1] * _I6
    xy, xz, yz = s[2] * _I2, s[3] * _I2, s[4] * _I2
    return [xx * p[0] + xy * p[1] + xz * p[2], xy * p[0] + yy * p[1] + yz * p[2], xz * p[0] + yz * p[1] + zz * p[2]]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


# Real-space scalars: derivatives of the shell / ball convolutions of the screened Green's function.
_GLX, _GLW = np.polynomial.legendre.leggauss(64)


def _kernel(k, s, d=0):
    """Convolution kernel (shell-shell, shell-ball, ball-ball) on [-2, 2], and its right derivatives."""
    t = np.abs(s)
    c = [np.array([2.0, -1.0]) / 4, np.array([4.0, 0.0, -3.0, 1.0]) / 8,
         3 * np.array([32.0, 0.0, -40.0, 20.0, 0.0, -1.0]) / 160][k]
    for _ in range(d):
        c = c[1:] * np.arange(1, len(c))
    v = sum(cc * t ** i for i, cc in enumerate(c)) if len(c) else 0.0 * t
    return np.where(t <= 2.0 if d == 0 else t < 2.0, v, 0.0)


def _conv(k, n, r, xi):
    """n-th derivative of the convolved profile at r >= 0."""
    c, sp = 1.0 / (8.0 * math.pi), math.sqrt(math.pi)
    tot = np.zeros_like(r)
    rb = np.minimum(r, 2.0)
    for lo, hi in ((0 * r - 2.0, 0 * r), (0 * r, rb), (rb, 0 * r + 2.0)):
        half = 0.5 * (hi - lo)
        s = (0.5 * (hi + lo))[:, None] + half[:, None] * _GLX
        t = r[:, None] - s
        E, g, u = torch.erf(torch.from_numpy(xi * t)).numpy(), np.exp(-(xi * t) ** 2), (xi * t) ** 2
        f = c * [t * t * E + t * g / (xi * sp), 2 * t * E + g / (xi * sp), 2 * E + 2 * xi / sp * t * g,
                 2 * xi / sp * g * (3 - 2 * u), 4 * xi ** 3 / sp * t * g * (2 * u - 5),
                 4 * xi ** 3 / sp * g * (-4 * u * u + 16 * u - 5)][n]
        if n <= 2:
            f = f - c * [t * np.abs(t), 2 * np.abs(t), 2 * np.sign(t)][n]
        tot += half * np.sum(_GLW * _kernel(k, s) * f, 1)
    return tot - 4 * c * _kernel(k, r, n - 3) if n >= 3 else tot


def _scalars(r, xi):
    """The 7 translation-stresslet scalars and the 3 rotation scalars at r (array)."""
    phi, psi = {}, {}
    for k in range(3):
        U = [_conv(k, n, r, xi) for n in range(5)]
        psi[k] = (None, U[1] / r - U[0] / r ** 2, U[2] / r - 2 * U[1] / r ** 2 + 2 * U[0] / r ** 3,
                  U[3] / r - 3 * U[2] / r ** 2 + 6 * U[1] / r ** 3 - 6 * U[0] / r ** 4,
                  U[4] / r - 4 * U[3] / r ** 2 + 12 * U[2] / r ** 3 - 24 * U[1] / r ** 4 + 24 * U[0] / r ** 5)
        V = [-U[2], -U[3], -U[4]]
        phi[k] = (V[0] / r, V[1] / r - V[0] / r ** 2, V[2] / r - 2 * V[1] / r ** 2 + 2 * V[0] / r ** 3)
    ap = {k: psi[k][2] / r - psi[k][1] / r ** 2 for k in psi}
    d = {k: psi[k][3] - 3 * psi[k][2] / r + 3 * psi[k][1] / r ** 2 for k in psi}
    dp = psi[2][4] - 3 * psi[2][3] / r + 6 * psi[2][2] / r ** 2 - 6 * psi[2][1] / r ** 3
    return np.stack([phi[0][0] + psi[0][1] / r, phi[0][0] + psi[0][2], -(phi[1][1] + 2 * ap[1]), -d[1],
                     -(phi[2][1] / r + 2 * ap[2] / r), -(0.5 * (phi[2][2] - phi[2][1] / r) + 2 * d[2] / r),
                     -(dp - 3 * d[2] / r),
                     phi[1][1] / 2, -(phi[2][2] + phi[2][1] / r) / 4, (phi[2][2] - phi[2][1] / r) / 4])


class _Table:
    """Chebyshev fits of the scalars on [0.2, 2] and [2, rcut] (they have a kink at contact)."""

    def __init__(self, xi, rcut):
        self.parts = []
        for lo, hi, deg in ((0.2, 2.0, 16), (2.0, max(rcut, 2.1), 48)):
            x = np.cos(math.pi * (np.arange(deg + 1) + 0.5) / (deg + 1))
            f = _scalars(0.5 * (hi + lo) + 0.5 * (hi - lo) * x, xi)
            self.parts.append((lo, hi, np.polynomial.chebyshev.chebfit(x, f.T, deg)))
        z = np.zeros(1)
        self.uf = float(2.0 / 3.0 * -_conv(0, 3, z, xi)[0])
        u5 = float(_conv(2, 5, z, xi)[0])
        self.es, self.ol = u5 / 5.0, u5 / 6.0

    def at(self, r, which):
        out = []
        near = r < 2.0
        some = bool(near.any())
        for q in which:
            both = []
            for lo, hi, c in self.parts[0 if some else 1:]:
                x = (2 * r - (hi + lo)) / (hi - lo)
                x.clamp_(min=-1.4, max=1.0)
                b1, b2 = torch.zeros_like(r), torch.zeros_like(r)
                for cc in c[:0:-1, q]:
                    b1, b2 = 2 * x * b1 - b2 + float(cc), b1
                both.append(x * b1 - b2 + float(c[0, q]))
            out.append(torch.where(near, both[0], both[1]) if some else both[0])
        return out


class _Exact:
    """The split mobility of one configuration in FP64."""

    def __init__(self, rules, table, pos, index0=0, mode0=0):
        self.p, self.t, self.index0, self.mode0 = rules, table, index0, mode0
        p = rules
        self.A = torch.tensor(p.A, device='cuda')
        self.Ai = torch.linalg.inv(self.A)
        self.z = (pos.double() @ self.Ai.T) % p.L
        self._pairs()

    def _pairs(self):
        p, z, n = self.p, self.z, self.p.n
        nc = int(p.L * math.sqrt(p.lam_min) / p.rcut)
        if nc < 3:
            order, start, stencil = torch.arange(n, device='cuda'), None, None
        else:
            c = (z * (nc / p.L)).long().clamp_(max=nc - 1)
            order = torch.argsort((c[:, 0] * nc + c[:, 1]) * nc + c[:, 2])
            c = c[order]
            count = torch.bincount((c[:, 0] * nc + c[:, 1]) * nc + c[:, 2], minlength=nc ** 3)
            start = torch.cat([count.new_zeros(1), count.cumsum(0)])
            o = torch.arange(-1, 2, device='cuda')
            stencil = torch.stack(torch.meshgrid(o, o, o, indexing='ij'), -1).reshape(-1, 3)
        zs = z[order]
        I, J, D = [], [], []
        step = max(1, min(32768, (1 << 25) // n if start is None else 32768))
        for b in range(0, n, step):
            e = min(n, b + step)
            if start is None:
                i = torch.arange(b, e, device='cuda').repeat_interleave(n)
                j = torch.arange(n, device='cuda').repeat(e - b)
            else:
                q = (c[b:e, None, :] + stencil) % nc
                q = ((q[..., 0] * nc + q[..., 1]) * nc + q[..., 2]).reshape(-1)
                m = start[q + 1] - start[q]
                i = torch.arange(b, e, device='cuda').repeat_interleave(27).repeat_interleave(m)
                j = torch.arange(len(i), device='cuda') - (m.cumsum(0) - m - start[q]).repeat_interleave(m)
            d = zs[i] - zs[j]
            d = (d - p.L * torch.round(d / p.L)) @ self.A.T
            hit = ((d * d).sum(1) < p.rcut ** 2) & (i != j)
            I.append(order[i[hit]])
            J.append(order[j[hit]])
            D.append(d[hit])
        self.i, self.j, self.d = torch.cat(I), torch.cat(J), torch.cat(D)

    def real(self, v):
        """M_r v for v of width 8 ([F, S]) or 11 ([F, L, S])."""
        rot = v.shape[1] == 11
        o = v * torch.tensor([self.t.uf] * 3 + ([self.t.ol] * 3 if rot else []) + [self.t.es] * 5, dtype=torch.float64,
                             device='cuda')
        for b in range(0, len(self.i), 1 << 24):
            i, d = self.i[b:b + (1 << 24)], self.d[b:b + (1 << 24)]
            w = v[self.j[b:b + (1 << 24)]].T
            r = d.norm(dim=1)
            rh = list((d / r[:, None]).T)
            f = self.t.at(r, range(10 if rot else 7))
            F, s = w[:3], w[-5:]
            S = _s_mul(s, rh)
            q, rf = _dot(rh, S), _dot(rh, F)
            U = [f[0] * F[m] + (f[1] - f[0]) * rf * rh[m] + f[2] * S[m] + f[3] * q * rh[m] for m in range(3)]
            yf, ys, yr = _sym_y(F, rh), _sym_y(S, rh), _sym_y(rh, rh)
            E = [-0.5 * f[2] * yf[m] - 0.5 * f[3] * rf * yr[m] + f[4] * s[m] + f[5] * ys[m] + 0.5 * f[6] * q * yr[m]
                 for m in range(5)]
            O = []
            if rot:
                Lt = w[3:6]
                rl, xl, xf, sx = _dot(rh, Lt), _cross(rh, Lt), _cross(rh, F), _cross(S, rh)
                U = [U[m] + f[7] * xl[m] for m in range(3)]
                O = [f[7] * xf[m] + f[8] * Lt[m] + f[9] * rl * rh[m] + 2 * f[9] * sx[m] for m in range(3)]
                yl = _sym_y(xl, rh)
                E = [E[m] + f[9] * yl[m] for m in range(5)]
            o.index_add_(0, i, torch.stack(U + O + E, 1))
        return o

    def _support(self, b, e):
        """Flat grid indices and Gaussian weights of the supports of particles b..e."""
        p, z = self.p, self.z[b:e]
        if p.P % 2:
            i0 = torch.round(z / p.h) - (p.P - 1) // 2
        else:
            i0 = torch.floor(z / p.h) - p.P // 2 + 1
        g = i0[:, None, :] + torch.arange(p.P, device='cuda')[None, :, None]
        dx = g * p.h - z[:, None, :]
        g = g.long() % p.Ng
        idx = (g[:, :, None, None, 2] * p.Ng + g[:, None, :, None, 1]) * p.Ng + g[:, None, None, :, 0]
        G = (self.A.T @ self.A).tolist()
        X, Y, Z = dx[:, None, None, :, 0], dx[:, None, :, None, 1], dx[:, :, None, None, 2]
        al = 2 * p.xi ** 2 / p.eta
        qf = G[0][0] * X * X + G[1][1] * Y * Y + G[2][2] * Z * Z + 2 * (G[0][1] * X * Y + G[0][2] * X * Z + G[1][2] * Y * Z)
        return idx.reshape(e - b, -1), ((al / math.pi) ** 1.5 * torch.exp(-al * qf)).reshape(e - b, -1)

    def _chunks(self):
        step = max(1, (1 << 25) // self.p.P ** 3)
        return [(b, min(self.p.n, b + step)) for b in range(0, self.p.n, step)]

    def _modes(self):
        """Wave vectors, their shape factors and the modes that count, on the half spectrum [z][y][x]."""
        p, h = self.p, self.p.Ng // 2
        m = torch.arange(p.Ng, device='cuda')
        s = torch.where(m <= h, m, m - p.Ng).double()
        mz, my, mx = torch.meshgrid(s, s, s[:h + 1], indexing='ij')
        B = (2 * math.pi / p.L * self.Ai.T).tolist()
        k = [B[d][0] * mx + B[d][1] * my + B[d][2] * mz for d in range(3)]
        live = (mx != h) & (my != h) & (mz != h) & ((mx != 0) | (my != 0) | (mz != 0))
        k2 = torch.where(live, _dot(k, k), 1.0)
        kk = torch.sqrt(k2)
        s0 = torch.sin(kk) / kk
        small = kk < 0.1
        x2 = k2
        s1 = torch.where(small, 1 / 3 - x2 / 30 + x2 ** 2 / 840 - x2 ** 3 / 45360 + x2 ** 4 / 3991680,
                         (torch.sin(kk) - kk * torch.cos(kk)) / (kk * k2))
        return k, k2, s0, s1, live

    def _interp(self, modes, u, rot=False):
        """Velocities, (rotations and) strains at the particles from the velocity modes u."""
        p = self.p
        k, _, s0, s1, live = modes
        u = [torch.where(live, w, 0.0) for w in u]
        g = [s0 * w for w in u]
        if rot:
            g += [-1.5j * s1 * w for w in _cross(u, k)]
        g += [1.5j * s1 * w for w in _sym_y(u, k)]
        sig = p.V / float(p.Ng) ** 3
        o = torch.empty((p.n, len(g)), dtype=torch.float64, device='cuda')
        grids = []
        for q in g:
            grids.append(torch.fft.irfftn(q, s=(p.Ng,) * 3, norm='forward').reshape(-1))
        for b, e in self._chunks():
            idx, w = self._support(b, e)
            for m, q in enumerate(grids):
                o[b:e, m] = (w * q[idx]).sum(1)
        return o, sig

    def wave(self, v):
        p = self.p
        rot = v.shape[1] == 11
        grid = torch.zeros((v.shape[1], p.Ng ** 3), dtype=torch.float64, device='cuda')
        for b, e in self._chunks():
            idx, w = self._support(b, e)
            for m in range(v.shape[1]):
                grid[m].index_add_(0, idx.reshape(-1), (w * v[b:e, m, None]).reshape(-1))
        spec = [torch.fft.rfftn(q.reshape((p.Ng,) * 3)) for q in grid]
        del grid
        modes = self._modes()
        k, k2, s0, s1, _ = modes
        sk = _s_mul(spec[-5:], k)
        f = [s0 * spec[m] - 3j * s1 * sk[m] for m in range(3)]
        if rot:
            kl = _cross(k, spec[3:6])
            f = [f[m] + 1.5j * s1 * kl[m] for m in range(3)]
        u = k2 / (4 * p.xi ** 2)
        c = (1 + u) * torch.exp(-(1 - p.eta) * u) / k2 / p.V
        fk = _dot(k, f) / k2
        o, sig = self._interp(modes, [c * (f[m] - k[m] * fk) for m in range(3)], rot)
        return o * sig * sig

    def apply(self, v):
        return self.real(v) + self.wave(v)

    def lanczos(self, z):
        V, al, be, prev = [z / z.norm()], [], [], None
        for j in range(100):
            w = self.real(V[j])
            h = torch.zeros(j + 1, dtype=torch.float64, device='cuda')
            for _ in range(2):
                c = torch.stack([(q * w).sum() for q in V])
                for q, cc in zip(V, c):
                    w = w - cc * q
                h += c
            al.append(float(h[j]))
            T = np.diag(al) + np.diag(be, 1) + np.diag(be, -1)
            lam, Q = np.linalg.eigh(T)
            c = Q @ (np.sqrt(np.maximum(lam, 0)) * Q[0])
            if j and np.linalg.norm(c - np.append(prev, 0.0)) / np.linalg.norm(c) <= self.p.tol:
                break
            prev = c
            be.append(float(w.norm()))
            V.append(w / be[-1])
        return float(z.norm()) * sum(cc * q for cc, q in zip(c.tolist(), V))

    def sample(self, seed, counter):
        """Unscaled Brownian velocities M_r^{1/2} w1 + M_w^{1/2} dW2, in-kernel streams 1 and 2."""
        p = self.p
        w1 = _normals(seed, counter, 1, 8 * self.index0 + torch.arange(8 * p.n, device='cuda'))[0].reshape(-1, 8)
        y = self.lanczos(w1)
        h, nk = p.Ng // 2, p.Ng ** 2 * (p.Ng // 2 + 1)
        modes = self._modes()
        k, k2 = modes[:2]
        m = torch.arange(p.Ng, device='cuda')
        mz, my, mx = torch.meshgrid(m, m, m[:h + 1], indexing='ij')
        twin = (mx == 0) & ((mz > h) | ((mz == 0) & (my > h)))
        src = torch.where(twin, (-mz) % p.Ng * p.Ng + (-my) % p.Ng, mz * p.Ng + my) * (h + 1) + mx
        d = []
        for q in range(3):
            re, im = _normals(seed, counter, 2, 3 * self.mode0 + q * nk + src)
            d.append(torch.complex(re, torch.where(twin, -im, im)) * _I2)
        u = k2 / (4 * p.xi ** 2)
        c = torch.sqrt((1 + u) / k2 / p.V) * torch.exp(-0.5 * (1 - p.eta) * u)
        dk = _dot(k, d) / k2
        o, sig = self._interp(modes, [c * (d[m] - k[m] * dk) for m in range(3)])
        return y + o * sig

    def solve(self, b):
        """S with M_ES S = b (GMRES to the relative residual tol)."""
        beta = float(b.norm())
        if beta == 0.0:
            return torch.zeros_like(b)
        V, H, zero = [b / beta], np.zeros((51, 50)), torch.zeros((self.p.n, 3), dtype=torch.float64, device='cuda')
        for j in range(50):
            w = self.apply(torch.cat([zero, V[j]], 1))[:, 3:]
            for _ in range(2):
                c = torch.stack([(q * w).sum() for q in V])
                for q, cc in zip(V, c):
                    w = w - cc * q
                H[:j + 1, j] += c.cpu().numpy()
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            e1 = np.eye(j + 2)[0] * beta
            y = np.linalg.lstsq(H[:j + 2, :j + 1], e1, rcond=None)[0]
            if np.linalg.norm(e1 - H[:j + 2, :j + 1] @ y) / beta <= self.p.tol:
                break
        return sum(float(c) * q for c, q in zip(y, V))

    def overlap(self):
        r = self.d.norm(dim=1)
        f = torch.where(r < 2.0, SPRING * (2.0 - r) / r, 0.0)
        o = torch.zeros((self.p.n, 3), dtype=torch.float64, device='cuda')
        return o.index_add_(0, self.i, f[:, None] * self.d)


def _normals(seed, step, stream, index):
    """Philox4x32-10 Box-Muller pairs for counter (index, step, stream) and key seed."""
    m32 = 0xFFFFFFFF
    c = [index & m32, index >> 32, torch.full_like(index, step & m32), torch.full_like(index, stream)]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57     # low 64 bits; the shifts below are masked
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u1, u2 = (c[0].double() + 0.5) * 2.0 ** -32, (c[1].double() + 0.5) * 2.0 ** -32
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


def _exact_step(x, rules, table, seed, step, overlap=False, index0=0, mode0=0):
    s, L = math.sqrt(2.0 / DT), rules.L
    at = _Exact(rules, table, x, index0, mode0)
    F = at.overlap() if overlap else None
    B = s * at.sample(seed, step)
    at = _Exact(rules, table, (x + 0.5 * DT * B[:, :3]) % L, index0, mode0)
    v = torch.zeros_like(B)
    b = -B[:, 3:]
    if overlap:
        v[:, :3] = F
        b = b - at.apply(v)[:, 3:]
    v[:, 3:] = at.solve(b)
    out = (x + DT * (B + at.apply(v))[:, :3]) % L, v[:, 3:].contiguous()
    return out + (F,) if overlap else out


def _exact_rfd(x, rules, table, seed, step, delta=1e-3):
    def constrained(at, b, F):
        v = torch.zeros((rules.n, 8), dtype=torch.float64, device='cuda')
        if F is not None:
            v[:, :3] = F
            b = b - at.apply(v)[:, 3:]
        v[:, 3:] = at.solve(b)
        return at.apply(v)[:, :3], v[:, 3:].contiguous()
    at = _Exact(rules, table, x)
    B = math.sqrt(2.0 / DT) * at.sample(seed, step)
    U, S = constrained(at, -B[:, 3:], None)
    W = _normals(seed, step, 3, torch.arange(3 * rules.n, device='cuda'))[0].reshape(-1, 3)
    R = [constrained(_Exact(rules, table, (x + sgn * 0.5 * delta * W) % rules.L), 0.0, W)[0] for sgn in (1, -1)]
    return (x + DT * (B[:, :3] + U + (R[0] - R[1]) / delta)) % rules.L, S


def exact(case, seed):
    ins, call = _inputs(case, seed), case['call']
    out, index0, mode0, table = [], 0, 0, None
    for q, i in enumerate(ins):
        p = _Rules(i['n'], i['L'], case['xi'], case['tol'], _deform(case))
        table = table or _Table(p.xi, p.rcut)
        kind = _KINDS[q % 3] if call == 'serve' else call
        step = q if call == 'serve' else 1
        if kind in ('mobility', 'mobility11'):
            v = torch.cat([i['F'], i['Lt'], i['S']] if kind == 'mobility11' else [i['F'], i['S']], 1).double()
            o = _Exact(p, table, i['pos']).apply(v)
            out.append([o[:, b:e].contiguous() for b, e in (((0, 3), (3, 6), (6, 11)) if kind == 'mobility11' else ((0, 3), (3, 8)))])
        elif kind == 'sample':
            o = math.sqrt(2.0 / DT) * _Exact(p, table, i['pos']).sample(seed, step)
            out.append([o[:, :3].contiguous(), o[:, 3:].contiguous()])
        elif kind == 'rfd':
            out.append(_exact_rfd(i['pos'], p, table, seed, step))
        else:
            at = (index0, mode0) if call == 'batch' else (0, 0)
            out.append(_exact_step(i['pos'], p, table, seed, step, case['overlap'] > 0, *at))
        index0 += i['n']
        mode0 += p.Ng ** 2 * (p.Ng // 2 + 1)
    if call == 'serve':
        return out
    if call == 'batch':
        return [torch.cat([o[m] for o in out]) for m in (0, 1)]
    return out[0]
