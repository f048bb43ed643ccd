"""The work a user has this library do, as measurable cases.

Every case is one pass through the public entry points (the ctypes binding of
include/mgmlmc.h) on device buffers, at sizes of this repository's tests and
benchmark or generic ones.  Kinds:

* dslash    the Wilson operator D on the fine lattice (FP32 in the canonical
            or the internal order, FP64, BF16 storage)
* sap       the fine-level smoother: red/black Schwarz sweeps from zero
* coarse    the Galerkin stencil D_1 = P^H D P on the first coarse lattice
* transfer  restriction P^H of a fine vector and prolongation P of a coarse
            one, the two halves of a coarse-grid correction
* net       forward pass of the learned gauge-covariant network
* netgrad   its loss and weight gradient (what a training loop calls)
* solve     D z = b to 1e-12 by multigrid-preconditioned FGMRES
* build     the set-up phase on a new gauge field: rough test vectors, P_l,
            D_{l+1}, the dense coarsest inverse; then first operator calls
* estimate  every term of the orthogonal multilevel estimator of tr(D^-1)

exact() restates each in plain complex128 torch (no code of this repository).
Vectors there are [rhs, t, z, y, x, dof], links [t, z, y, x, mu, 3, 3].
"""
import math

import numpy as np
import torch

from paper_2509_11424_gb300 import mgmlmc as M

EPS, MASS = 0.4, -0.40  # spread of the synthetic links and bare mass of the benchmark's ensembles
TOL = 1e-12


def _case(name, kind, dims, **kw):
    c = {'name': name, 'kind': kind, 'Lx': dims[0], 'Ly': dims[1], 'Lz': dims[2], 'Lt': dims[3]}
    c.update(kw)
    return c


def listed():
    return [
        # one operator call on the smallest lattice of the tests, caller's own layout: launch latency
        _case('dslash_f32_8x8x8x8', 'dslash', (8, 8, 8, 8), prec='f32', internal=False, nrhs=1),
        # the Krylov operator inside a mixed solve: the benchmark's 32^4, a block of 4 right-hand sides
        _case('dslash_f32_32x32x32x32', 'dslash', (32, 32, 32, 32), prec='f32', internal=True, nrhs=4),
        # the true-residual operator of every solve, FP64, an odd number of right-hand sides
        _case('dslash_f64_24x24x24x24', 'dslash', (24, 24, 24, 24), prec='f64', internal=False, nrhs=3),
        # the smoother of the fine level, where a solve spends most of its time
        _case('sap_f32_32x32x32x32', 'sap', (32, 32, 32, 32), prec='f32', internal=True, nrhs=4, sweeps=2, iters=4),
        # the same on a ragged lattice: 2^4 blocks, one right-hand side, caller's own layout
        _case('sap_f32_12x12x12x20', 'sap', (12, 12, 12, 20), prec='f32', internal=False, nrhs=1, sweeps=1, iters=4),
        # coarse operator in the K-cycle (FP32) and as the true residual of the coarse solves (FP64)
        _case('coarse_f32_24x24x24x48', 'coarse', (24, 24, 24, 48), prec='f32', block=4, ntv=16, nrhs=4),
        _case('coarse_f64_16x16x16x32', 'coarse', (16, 16, 16, 32), prec='f64', block=4, ntv=16, nrhs=8),
        # the transfers of a coarse-grid correction
        _case('transfer_f32_24x24x24x48', 'transfer', (24, 24, 24, 48), prec='f32', block=4, ntv=16, nrhs=4),
        # the learned network with the default number of channels, and a training gradient
        _case('net_f32_16x16x16x16', 'net', (16, 16, 16, 16), prec='f32', channels=16, nrhs=2),
        _case('netgrad_f64_8x8x8x8', 'netgrad', (8, 8, 8, 8), channels=4, nrhs=4),
        # whole calls: the mixed-precision solve and the set-up of the 16^4 workload
        _case('solve_mixed_16x16x16x16', 'solve', (16, 16, 16, 16), prec='f32', ntv=16, nrhs=8),
        _case('build_f64_16x16x16x16', 'build', (16, 16, 16, 16), ntv=16, rounds=3, iters=20),
    ]


# ---------------------------------------------------------------- drawing
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, step, lo, hi, vmax):
    """Four extents, multiples of step in lo .. hi, with at most vmax sites."""
    while True:
        d = [step * max(1, int(round(_log_int(rng, lo, hi) / step))) for _ in range(4)]
        if min(d) >= max(2, lo) and d[0] * d[1] * d[2] * d[3] <= vmax:
            return d


def draw(rng):
    kind = rng.choice(['dslash', 'dslash', 'sap', 'sap', 'coarse', 'coarse', 'transfer', 'net', 'netgrad', 'solve',
                       'build', 'estimate'])
    if kind == 'dslash':
        prec = rng.choice(['f32', 'f32', 'f64', 'bf16'])
        d = _dims(rng, rng.choice([1, 2, 4]), 4, 40, 32 ** 4 if prec != 'f64' else 24 ** 4)
        c = dict(prec=prec, internal=prec != 'f64' and rng.random() < 0.5, nrhs=_log_int(rng, 1, 4))
    elif kind == 'sap':
        prec = rng.choice(['f32', 'f32', 'f32', 'f64'])
        d = _dims(rng, rng.choice([4, 8, 8, 16]), 8, 32, 32 ** 4 if prec == 'f32' else 16 ** 4)
        c = dict(prec=prec, internal=prec == 'f32' and rng.random() < 0.5, nrhs=_log_int(rng, 1, 4),
                 sweeps=rng.choice([1, 2]), iters=rng.choice([2, 3, 4]))
    elif kind in ('coarse', 'transfer'):
        prec = rng.choice(['f32', 'f32', 'f64'])
        b = rng.choice([2, 3, 4, 4])
        ntv = rng.choice([8, 12, 16, 16, 16, 20, 24])
        # level 1 holds at most the listed cases' blocks (2592 sites of 32 dofs)
        vmax = min((24 ** 3 * 48) // 4 if prec == 'f64' else 24 ** 3 * 48, int(2592 * (16 / ntv) ** 2) * b ** 4)
        d = _dims(rng, 2 * b, 2 * b, 48, vmax)
        c = dict(prec=prec, block=b, ntv=ntv, nrhs=_log_int(rng, 1, 4 if prec == 'f32' else 8))
        if kind == 'coarse' and prec == 'f32' and d[0] * d[1] * d[2] * d[3] * 8 <= vmax:
            c['nrhs'] = _log_int(rng, 4, 32)
    elif kind == 'net':
        prec = rng.choice(['f32', 'f32', 'f64'])
        ch = rng.choice([1, 1, 2, 3, 4, 8, 16]) if prec == 'f32' else rng.choice([1, 2])
        d = _dims(rng, rng.choice([1, 2, 4]), 4, 24, 16 ** 4)
        c = dict(prec=prec, channels=ch, nrhs=_log_int(rng, 1, 2))
    elif kind == 'netgrad':
        d = _dims(rng, rng.choice([1, 2, 4]), 4, 10, 8 ** 4)
        c = dict(channels=rng.choice([1, 2, 3, 4]), nrhs=_log_int(rng, 1, 4))
    elif kind == 'solve':
        prec = rng.choice(['f32', 'f32', 'f64'])
        d = _dims(rng, 8, 8, 16, 16 ** 4 if prec == 'f32' else 8 ** 4 * 2)
        c = dict(prec=prec, ntv=rng.choice([8, 12, 16]), nrhs=_log_int(rng, 1, 8))
    elif kind == 'build':
        d = _dims(rng, 8, 8, 16, 16 ** 4)
        c = dict(ntv=rng.choice([8, 12, 16]), rounds=rng.choice([1, 2, 3]), iters=rng.choice([10, 15, 20]))
    else:
        d = _dims(rng, 8, 8, 16, 8 ** 3 * 16)
        c = dict(ntv=rng.choice([8, 12, 16]), samples=_log_int(rng, 1, 4))
    c = _case('', kind, d, **c)
    del c['name']
    return c


# ---------------------------------------------------------------- inputs
def _geo(case):
    return [case['Lx'], case['Ly'], case['Lz'], case['Lt']]


def _volume(case):
    return case['Lx'] * case['Ly'] * case['Lz'] * case['Lt']


def _gen(seed):
    g = torch.Generator(device='cuda')
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape):
    re = torch.randn(*shape, generator=g, device='cuda', dtype=torch.float64)
    im = torch.randn(*shape, generator=g, device='cuda', dtype=torch.float64)
    return torch.complex(re, im) * math.sqrt(0.5)


def _mul3(a, b):
    return sum(a[:, :, k, None] * b[:, k, None, :] for k in range(3))


def _links(dims, seed):
    """SU(3) links exp(i EPS H), H random traceless Hermitian, [t, z, y, x, mu, 3, 3]."""
    g = _gen(seed)
    n = 4 * dims[0] * dims[1] * dims[2] * dims[3]
    eye = torch.eye(3, dtype=torch.complex128, device='cuda')
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device='cuda')
    step = 1 << 20
    for a in range(0, n, step):
        A = _normal(g, min(step, n - a), 3, 3)
        H = 0.5 * (A + A.conj().transpose(1, 2))
        H = H - (torch.einsum('naa->n', H).real / 3.0)[:, None, None] * eye
        X = H * (1j * EPS / 16.0)
        E = eye + X / 14.0
        for k in range(13, 0, -1):
            E = eye + _mul3(X, E) / k
        for _ in range(4):
            E = _mul3(E, E)
        out[a:a + step] = E
    return out.view(dims[3], dims[2], dims[1], dims[0], 4, 3, 3)


class _Context:
    """A library context that is given back with its last user."""

    def __init__(self, dims):
        self.handle = M.mgmlmc_create(dims, torch.cuda.current_stream())

    def __del__(self):
        if getattr(self, 'handle', None):
            M.mgmlmc_destroy(self.handle)
            self.handle = None


def _context(case, U):
    c = _Context(_geo(case))
    M.mgmlmc_set_gauge(c.handle, U.view(-1), on_device=True)
    M.mgmlmc_set_mass(c.handle, MASS)
    return c


SOLVER = dict(tol=TOL, restart=24, max_iter=2000, smoother=M.SMOOTHER_SAP, smoother_steps=1, sap_iters=4,
              coarse_iters=4, inner_tol=1e-6, coarse_smoother_steps=4)
LEVELS = [(4, 4, 4, 4), (2, 2, 2, 2)]  # aggregates of the 16^4 workload


def _hierarchy(case):
    """Aggregates and test-vector counts of a three-level hierarchy on the case's lattice."""
    if case['kind'] not in ('coarse', 'transfer'):
        return LEVELS, [case['ntv'], case['ntv']]
    # the last level only closes the hierarchy: the largest aggregates the library takes (48 KB of rows)
    ntv = case['ntv']
    b = [L // case['block'] for L in _geo(case)]
    lat = list(b)
    while b[0] * b[1] * b[2] * b[3] * ntv * 16 > 48 * 1024:
        i = b.index(max(b))
        b[i] = max(k for k in range(1, b[i]) if lat[i] % k == 0)
    return [(case['block'],) * 4, tuple(b)], [ntv, min(8, ntv)]


def _weights(channels, seed):
    """Network weights in the library's order, complex128 on the host: small, with a Jacobi step on channel 0."""
    r = np.random.default_rng(seed)
    out = []
    for cin, cout, s in ((1, channels, 1.0), (channels, channels, 1.0), (channels, 1, 1.0 / (4.0 + MASS))):
        w = 0.05 * (r.standard_normal((9, cout, cin, 4, 4)) + 1j * r.standard_normal((9, cout, cin, 4, 4)))
        w[0, 0, 0] += s * np.eye(4)
        out.append(w)
    return out


def _vectors(case, seed, n):
    return _normal(_gen(seed * 2 + 1), case['nrhs'], n)


def prepare(case, seed):
    kind, dims = case['kind'], _geo(case)
    n = 12 * _volume(case)
    U = _links(dims, seed * 2)
    ctx = _context(case, U)
    h = ctx.handle
    st = {'case': case, 'ctx': ctx, 'seed': seed}
    prec = {'f32': M.FP32, 'f64': M.FP64, 'bf16': M.BF16}[case.get('prec', 'f64')]
    st['prec'] = prec
    dt = torch.complex64 if prec == M.FP32 else torch.complex128
    if kind in ('dslash', 'sap'):
        if kind == 'sap':
            M.mgmlmc_set_solver(h, smoother=M.SMOOTHER_SAP, smoother_steps=case['sweeps'], sap_iters=case['iters'])
        x = _vectors(case, seed, n)
        if prec == M.BF16:
            x = torch.view_as_real(x).reshape(case['nrhs'], 2 * n).to(torch.bfloat16)
        else:
            x = x.to(dt)
        if case['internal']:
            xi = torch.empty_like(x)
            (M.mgmlmc_reorder_bf16 if prec == M.BF16 else M.mgmlmc_reorder)(h, x, xi, case['nrhs'], 1)
            x = xi
        st['op'] = (M.OP_D if kind == 'dslash' else M.OP_SMOOTH) | (M.LAYOUT_INTERNAL if case['internal'] else 0)
        st['x'], st['y'] = x, torch.empty_like(x)
    elif kind in ('coarse', 'transfer'):
        blocks, ntv = _hierarchy(case)
        M.mgmlmc_build_hierarchy(h, M.mg_params(blocks, ntv, setup_rounds=0, seed=seed))
        nc = M.mgmlmc_level_info(h, 1)[2]
        st['xc'] = _vectors(case, seed, nc).to(dt)
        if kind == 'coarse':
            st['yc'] = torch.empty_like(st['xc'])
        else:
            st['x'] = _normal(_gen(seed * 2 + 5), case['nrhs'], n).to(dt)
            st['y'], st['yc'] = torch.empty_like(st['x']), torch.empty_like(st['xc'])
    elif kind in ('net', 'netgrad'):
        M.mgmlmc_learned_init(h, case['channels'], 5000)
        w = np.concatenate([a.reshape(-1) for a in _weights(case['channels'], seed)])
        M.mgmlmc_learned_weights(h, w.view(np.float64).copy(), 1)
        st['x'] = _vectors(case, seed, n).to(dt)
        if kind == 'net':
            st['y'] = torch.empty_like(st['x'])
        else:
            st['grad'] = np.zeros(2 * w.size)
    elif kind == 'solve':
        M.mgmlmc_set_solver(h, precision=prec, **SOLVER)
        blocks, ntv = _hierarchy(case)
        M.mgmlmc_build_hierarchy(h, M.mg_params(blocks, ntv, setup_rounds=3, setup_iters=20, seed=seed))
        st['x'] = _vectors(case, seed, n)
        st['y'] = torch.empty_like(st['x'])
    elif kind == 'build':
        blocks, ntv = _hierarchy(case)
        st['params'] = M.mg_params(blocks, ntv, setup_rounds=case['rounds'], setup_iters=case['iters'], seed=seed)
        # what the first calls after the set-up act on
        size = [_level_size(case, l) for l in range(3)]
        st['x'] = [_normal(_gen(seed * 2 + 7 + l), 2, size[l]) for l in range(3)]
        st['y'] = [torch.empty(2, k, dtype=torch.complex128, device='cuda') for k in (size[1], size[2], size[1], size[0])]
    else:
        # the hierarchy from an FP64 set-up (a function of the inputs to 64-bit accuracy), then the mixed solver
        blocks, ntv = _hierarchy(case)
        M.mgmlmc_build_hierarchy(h, M.mg_params(blocks, ntv, setup_rounds=2, setup_iters=12, seed=seed))
        M.mgmlmc_set_solver(h, precision=M.FP32, **SOLVER)
        st['est'] = M.est_params(M.EST_ORTHOGONAL, [case['samples']] * 5, batch=case['samples'], seed=seed)
    return st


def _level_size(case, l):
    blocks, ntv = _hierarchy(case)
    v, dof = _volume(case), 12
    for i in range(l):
        v //= blocks[i][0] * blocks[i][1] * blocks[i][2] * blocks[i][3]
        dof = 2 * ntv[i]
    return v * dof


# ---------------------------------------------------------------- one pass
def run(st):
    case, h = st['case'], st['ctx'].handle
    kind, r = case['kind'], case.get('nrhs')
    if kind in ('dslash', 'sap'):
        M.mgmlmc_apply(h, st['op'], 0, st['prec'], st['x'], st['y'], r)
        return st['y']
    if kind == 'coarse':
        M.mgmlmc_apply(h, M.OP_D, 1, st['prec'], st['xc'], st['yc'], r)
        return st['yc']
    if kind == 'transfer':
        M.mgmlmc_apply(h, M.OP_RESTRICT, 0, st['prec'], st['x'], st['yc'], r)
        M.mgmlmc_apply(h, M.OP_PROLONG, 0, st['prec'], st['xc'], st['y'], r)
        return [st['yc'], st['y']]
    if kind == 'net':
        M.mgmlmc_apply(h, M.OP_NET, 0, st['prec'], st['x'], st['y'], r)
        return st['y']
    if kind == 'netgrad':
        loss = M.mgmlmc_learned_loss_grad(h, st['x'], r, st['grad'])
        return [loss, st['grad']]
    if kind == 'solve':
        M.mgmlmc_apply(h, M.OP_SOLVE, 0, M.FP64, st['x'], st['y'], r)
        return st['y']
    if kind == 'build':
        M.mgmlmc_build_hierarchy(h, st['params'])
        x, y = st['x'], st['y']
        M.mgmlmc_apply(h, M.OP_D, 1, M.FP64, x[1], y[0], 2)
        M.mgmlmc_apply(h, M.OP_D, 2, M.FP64, x[2], y[1], 2)
        M.mgmlmc_apply(h, M.OP_RESTRICT, 0, M.FP64, x[0], y[2], 2)
        M.mgmlmc_apply(h, M.OP_PROLONG, 0, M.FP64, x[1], y[3], 2)
        tr = M.mgmlmc_coarsest_trace(h)
        return y + [np.array([tr.real, tr.imag])]
    terms = M.mgmlmc_estimate_trace(h, st['est'])
    return [M.mgmlmc_last_samples(h, i, case['samples']) for i in range(len(terms))]


# ---------------------------------------------------------------- necessary work
def _net_flops(channels):
    c = channels
    return sum(9 * (ci * 288 + ci * co * 384) for ci, co in ((1, c), (c, c), (c, 1)))


def work(case):
    kind, V, r = case['kind'], _volume(case), case.get('nrhs', 1)
    es = {'f32': 8, 'f64': 16, 'bf16': 4}[case.get('prec', 'f64')]
    if kind == 'dslash':
        return {'bytes': V * (24 * r + 36) * es, 'flops': 1368 * V * r}
    if kind == 'sap':
        return {'bytes': V * (24 * r + 36) * es, 'flops': V * r * case['sweeps'] * (1368 * case['iters'] + 684)}
    if kind == 'coarse':
        Vc, m = V // case['block'] ** 4, 2 * case['ntv']
        return {'bytes': Vc * (9 * m * m + 2 * m * r) * es, 'flops': 72 * m * m * Vc * r}
    if kind == 'transfer':
        n, nc = 12 * V, V // case['block'] ** 4 * 2 * case['ntv']
        return {'bytes': 2 * (n * case['ntv'] + (n + nc) * r) * es, 'flops': 2 * 8 * n * case['ntv'] * r}
    if kind == 'net':
        return {'bytes': V * (24 * r + 36) * es, 'flops': V * r * _net_flops(case['channels'])}
    if kind == 'netgrad':
        return {'bytes': V * (12 * r + 36) * 16, 'flops': V * r * (3 * _net_flops(case['channels']) + 2 * 1368)}
    if kind == 'solve':  # right-hand sides in, solutions out; at least one application of D for each
        return {'bytes': V * (24 * r + 36) * 16, 'flops': 1368 * V * r}
    if kind == 'build':  # links in; the GMRES operators of the test vectors, P^H D P
        n, k = 12 * V, case['ntv']
        return {'bytes': (36 * V + 2 * k * n) * 16,
                'flops': 1368 * V * k * (case['rounds'] * case['iters'] + 2) + 8 * n * k * 2 * k * 3}
    return {'bytes': V * (36 + 24 * case['samples']) * 16, 'flops': 2 * 1368 * V * case['samples']}


# ---------------------------------------------------------------- 64-bit values
def _gamma():
    s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    out = []
    for B in [-1j * x for x in s] + [np.eye(2)]:
        g = np.zeros((4, 4), dtype=complex)
        g[:2, 2:] = B
        g[2:, :2] = B.conj().T
        out.append(torch.from_numpy(g).cuda())
    return out


def _shift(v, mu, fwd):
    """v(x + mu) (fwd) or v(x - mu) of a field [b, t, z, y, x, ...], antiperiodic in time."""
    ax = 4 - mu
    w = torch.roll(v, -1 if fwd else 1, ax)
    if mu == 3:
        w = w.clone()
        w[:, -1 if fwd else 0] *= -1
    return w


def _transport(v, U, mu, fwd):
    """U_mu(x) v(x + mu) or U_mu(x - mu)^H v(x - mu); v [b, t, z, y, x, spin, colour]."""
    Um = U[..., mu, :, :]
    if fwd:
        w, A = _shift(v, mu, True), Um
    else:
        w, A = _shift(v, mu, False), torch.roll(Um, 1, 3 - mu).conj().transpose(-1, -2)
    return sum(A[..., None, :, c] * w[..., c, None] for c in range(3))


def _edge(dims, b, mu, fwd):
    """1 where the hop in +-mu stays inside its block of extents b, [1, t, z, y, x, 1, 1]."""
    x = torch.arange(dims[mu], device='cuda')
    inside = ((x + 1) % b[mu] != 0) if fwd else (x % b[mu] != 0)
    shape = [1] * 7
    shape[4 - mu] = dims[mu]
    return inside.to(torch.float64).view(shape)


def _wilson(v, U, block=None):
    """D v; with `block` the hops that leave a block are dropped."""
    shape = v.shape
    dims = [shape[4], shape[3], shape[2], shape[1]]
    p = v.reshape(*shape[:5], 4, 3)
    out = (4.0 + MASS) * p
    for mu, g in enumerate(_gamma()):
        for fwd in (True, False):
            w = _transport(p, U, mu, fwd)
            gw = torch.einsum('st,bzyxwtc->bzyxwsc', g, w)
            hop = w - gw if fwd else w + gw
            if block is not None:
                hop = hop * _edge(dims, block, mu, fwd)
            out = out - 0.5 * hop
    return out.reshape(shape)


def _by_rhs(f, v, most=1 << 21):
    """f on a few right-hand sides at a time (bounded temporaries)."""
    k = max(1, most // max(1, v[0, ..., 0].numel()))
    return torch.cat([f(v[a:a + k]) for a in range(0, v.shape[0], k)])


def _field(x, dims):
    return x.reshape(x.shape[0], dims[3], dims[2], dims[1], dims[0], -1)


def _sap(b, U, block, sweeps, iters):
    dims = [b.shape[4], b.shape[3], b.shape[2], b.shape[1]]
    nb = [dims[i] // block[i] for i in range(4)]
    idx = [torch.arange(dims[i], device='cuda') // block[i] for i in range(4)]
    par = (idx[3][:, None, None, None] + idx[2][None, :, None, None] + idx[1][None, None, :, None]
           + idx[0][None, None, None, :]) % 2

    def blocksum(s):  # [rhs, t, z, y, x] -> the sum of each site's block at every site
        q = s.reshape(-1, nb[3], block[3], nb[2], block[2], nb[1], block[1], nb[0], block[0])
        q = q.sum(dim=(2, 4, 6, 8), keepdim=True).expand_as(q)
        return q.reshape(s.shape)

    z, r = torch.zeros_like(b), b.clone()
    for _ in range(sweeps):
        for colour in (0, 1):
            mask = (par == colour).to(torch.float64)[None, ..., None]
            rho, e = r * mask, torch.zeros_like(r)
            for _ in range(iters):
                q = _wilson(rho, U, block)
                num, den = blocksum((q.conj() * rho).sum(-1)), blocksum((q.abs() ** 2).sum(-1))
                al = torch.where(den > 1e-280, num / den.clamp_min(1e-280), torch.zeros_like(num))[..., None]
                e, rho = e + al * rho, rho - al * q
            z, r = z + e, r - _wilson(e, U)
    return z


def _sap_block(dims):
    for b in ((8, 4, 4, 2), (4, 4, 4, 4), (2, 2, 2, 2)):
        if all(L % k == 0 and (L // k) % 2 == 0 for L, k in zip(dims, b)):
            return b
    return None


class _Transfer:
    """P of one level: per aggregate and chirality the orthonormalised test vectors [k, t, z, y, x, dof]."""

    def __init__(self, tv, block):
        self.lat = [tv.shape[4], tv.shape[3], tv.shape[2], tv.shape[1]]
        self.block, self.half = block, tv.shape[5] // 2
        self.nc = [L // b for L, b in zip(self.lat, block)]
        A = self._blocks(tv).permute(1, 2, 3, 0)  # [X, c, row, k]
        for _ in range(2):  # Cholesky QR, twice
            G = A.conj().transpose(-1, -2) @ A
            L = torch.linalg.cholesky(G)
            A = torch.linalg.solve_triangular(L, A.conj().transpose(-1, -2), upper=False).conj().transpose(-1, -2)
        self.Q = A
        self.ntv = tv.shape[0]

    def _blocks(self, v):
        n, b = self.nc, self.block
        q = v.reshape(-1, n[3], b[3], n[2], b[2], n[1], b[1], n[0], b[0], 2, self.half)
        return q.permute(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10).reshape(v.shape[0], -1, 2, b[0] * b[1] * b[2] * b[3] * self.half)

    def restrict(self, v):
        y = torch.einsum('xcjk,rxcj->rxck', self.Q.conj(), self._blocks(v))
        return y.reshape(v.shape[0], self.nc[3], self.nc[2], self.nc[1], self.nc[0], 2 * self.ntv)

    def prolong(self, y):
        n, b = self.nc, self.block
        q = torch.einsum('xcjk,rxck->rxcj', self.Q, y.reshape(y.shape[0], -1, 2, self.ntv))
        q = q.reshape(-1, n[3], n[2], n[1], n[0], 2, b[3], b[2], b[1], b[0], self.half)
        q = q.permute(0, 1, 6, 2, 7, 3, 8, 4, 9, 5, 10)
        return q.reshape(y.shape[0], self.lat[3], self.lat[2], self.lat[1], self.lat[0], 2 * self.half)


def _z4(n, seed, sample0, term, count):
    """The library's documented Z4 noise (Philox4x64-10 by counter), [count, n] complex128."""
    vals = np.array([1, 1j, -1, -1j])
    out = np.empty((count, n), dtype=np.complex128)
    for k in range(count):
        start = (((sample0 + k) << 64) + (term << 128) - 1) % (1 << 256)
        bits = np.random.Philox(counter=start, key=int(seed)).random_raw(4 * ((n + 3) // 4))
        out[k] = vals[(bits[:n] >> np.uint64(62)).astype(np.int64)]
    return torch.from_numpy(out).cuda()


def _rough(D, v, iters):
    """argmin ||v - D w|| over the Krylov space of `iters` steps, normalised, for each vector."""
    shape, k = v.shape, v.shape[0]
    b = v.reshape(k, -1)
    beta = b.norm(dim=1)
    V = [b / beta[:, None]]
    H = torch.zeros(k, iters + 1, iters, dtype=torch.complex128, device='cuda')
    for i in range(iters):
        w = D(V[i].reshape(shape)).reshape(k, -1)
        for _ in range(2):
            for j in range(i + 1):
                h = (V[j].conj() * w).sum(1)
                H[:, j, i] += h
                w = w - h[:, None] * V[j]
        nw = w.norm(dim=1)
        H[:, i + 1, i] = nw
        V.append(w / nw[:, None])
    rhs = torch.zeros(k, iters + 1, 1, dtype=torch.complex128, device='cuda')
    rhs[:, 0, 0] = beta
    Qm, R = torch.linalg.qr(H)
    y = torch.linalg.solve_triangular(R, Qm.conj().transpose(-1, -2) @ rhs, upper=True)
    x = sum(y[:, j] * V[j] for j in range(iters))
    return (x / x.norm(dim=1)[:, None]).reshape(shape)


def _levels(case, seed, U, rounds, iters):
    """Operators D_l and transfers P_l of the hierarchy the library sets up."""
    dims = _geo(case)
    blocks, ntv = _hierarchy(case)
    D = [lambda v: _by_rhs(lambda w: _wilson(w, U), v)]
    P, lat, dof = [], dims, 12
    for l in range(2):
        n = lat[0] * lat[1] * lat[2] * lat[3] * dof
        tv = _field(_z4(n, seed, 0, 96 + l, ntv[l]), lat)
        for _ in range(rounds):
            tv = _rough(D[l], tv, iters)
        P.append(_Transfer(tv, blocks[l]))
        D.append(lambda v, p=P[l], d=D[l]: p.restrict(d(p.prolong(v))))
        lat, dof = [L // b for L, b in zip(lat, blocks[l])], 2 * ntv[l]
    return D, P, lat, dof


def _solve(D, b):
    """D x = b by BiCGStab in blocks of iterations, each restarted from the true residual."""
    shape, k = b.shape, b.shape[0]
    ap = lambda v: D(v.reshape(shape)).reshape(k, -1)  # noqa: E731
    dot = lambda a, c: (a.conj() * c).sum(1)[:, None]  # noqa: E731
    b = b.reshape(k, -1)
    x, bn = torch.zeros_like(b), b.norm(dim=1)
    for _ in range(12):
        r = b - ap(x)
        if float((r.norm(dim=1) / bn).max()) < 2e-15:
            break
        r0, p, rho = r.clone(), r.clone(), dot(r, r)
        goal = r.norm(dim=1) * 1e-7
        for _ in range(200):
            v = ap(p)
            al = rho / dot(r0, v)
            s = r - al * v
            t = ap(s)
            om = dot(t, s) / dot(t, t)
            x = x + al * p + om * s
            r = s - om * t
            new = dot(r0, r)
            if float((r.norm(dim=1) / goal).max()) < 1.0:
                break
            p = r + (new / rho) * (al / om) * (p - om * v)
            rho = new
    return x.reshape(shape)


def _dense(D, lat, dof):
    n = lat[0] * lat[1] * lat[2] * lat[3] * dof
    eye = torch.eye(n, dtype=torch.complex128, device='cuda')
    return torch.cat([D(_field(eye[a:a + 16], lat)).reshape(-1, n) for a in range(0, n, 16)]).transpose(0, 1)


def _layer(v, W, U):
    """phi[o] = sum_c sum_h W[h][o][c] T_h psi[c]; v [b, c, t, z, y, x, 4, 3]."""
    b, c = v.shape[:2]
    flat = v.reshape(b * c, *v.shape[2:])
    out = 0
    for h in range(9):
        t = flat if h == 0 else _transport(flat, U, (h - 1) // 2, h % 2 == 1)
        out = out + torch.einsum('ocst,bczyxwtq->bozyxwsq', W[h], t.reshape(v.shape))
    return out


def _net(x, Ws, U):
    v = x.reshape(x.shape[0], 1, *x.shape[1:5], 4, 3)
    for W in Ws:
        v = _layer(v, W, U)
    return v.reshape(x.shape)


def _soa(y, per):
    """[rhs, V, 12] to the library's internal order: chunks of `per` components over all sites."""
    r, V = y.shape[0], y.shape[1]
    return y.reshape(r, V, 12 // per, per).permute(0, 2, 1, 3).reshape(r, -1)


def exact(case, seed):
    kind, dims, V = case['kind'], _geo(case), _volume(case)
    n = 12 * V
    U = _links(dims, seed * 2)
    prec = case.get('prec', 'f64')
    if kind in ('dslash', 'sap'):
        x = _vectors(case, seed, n)
        if prec == 'bf16':
            x = torch.view_as_real(x).to(torch.bfloat16).to(torch.float64)
            x = torch.view_as_complex(x.contiguous())
            # the operator is that of the links as stored
            Ub = torch.view_as_real(U.to(torch.complex64).contiguous()).to(torch.bfloat16).to(torch.float64)
            U = torch.view_as_complex(Ub.contiguous())
        elif prec == 'f32':
            x = x.to(torch.complex64).to(torch.complex128)
        f = _field(x, dims)
        if kind == 'dslash':
            y = _by_rhs(lambda w: _wilson(w, U), f)
        else:
            block = _sap_block(dims)
            if block is None:
                return None
            y = _by_rhs(lambda w: _sap(w, U, block, case['sweeps'], case['iters']), f)
        y = y.reshape(case['nrhs'], V, 12)
        y = _soa(y, 4 if prec == 'bf16' else 2) if case['internal'] else y.reshape(case['nrhs'], n)
        return torch.view_as_real(y.contiguous()).reshape(case['nrhs'], 2 * n) if prec == 'bf16' else y
    if kind in ('coarse', 'transfer'):
        blocks, ntv = _hierarchy(case)
        P = _Transfer(_field(_z4(n, seed, 0, 96, ntv[0]), dims), blocks[0])
        lat = [L // b for L, b in zip(dims, blocks[0])]
        rnd = (lambda v: v.to(torch.complex64).to(torch.complex128)) if prec == 'f32' else (lambda v: v)
        nc = lat[0] * lat[1] * lat[2] * lat[3] * 2 * ntv[0]
        xc = _field(rnd(_vectors(case, seed, nc)), lat)
        if kind == 'coarse':
            return _by_rhs(lambda w: P.restrict(_wilson(P.prolong(w), U)), xc, 1 << 13).reshape(case['nrhs'], nc)
        x = _field(rnd(_normal(_gen(seed * 2 + 5), case['nrhs'], n)), dims)
        return [P.restrict(x).reshape(case['nrhs'], nc), P.prolong(xc).reshape(case['nrhs'], n)]
    if kind in ('net', 'netgrad'):
        x = _vectors(case, seed, n)
        if prec == 'f32':
            x = x.to(torch.complex64).to(torch.complex128)
        x = _field(x, dims)
        Ws = [torch.from_numpy(w).cuda() for w in _weights(case['channels'], seed)]
        if kind == 'net':
            return _by_rhs(lambda w: _net(w, Ws, U), x, 1 << 17).reshape(case['nrhs'], n)
        Ws = [w.requires_grad_(True) for w in Ws]
        d = x - _wilson(_net(x, Ws, U), U)
        loss = ((d.abs() ** 2).flatten(1).sum(1) / (x.abs() ** 2).flatten(1).sum(1)).sum()
        loss.backward()
        g = torch.cat([w.grad.reshape(-1) for w in Ws]).resolve_conj() * 0.5  # dL/dW*
        return [float(loss), torch.view_as_real(g).reshape(-1)]
    if kind == 'solve':
        b = _field(_vectors(case, seed, n), dims)
        return _by_rhs(lambda w: _solve(lambda v: _wilson(v, U), w), b, 1 << 20).reshape(case['nrhs'], n)
    if kind == 'build':
        D, P, lat, dof = _levels(case, seed, U, case['rounds'], case['iters'])
        lats = [dims, P[0].nc, P[1].nc]
        x = [_field(_normal(_gen(seed * 2 + 7 + l), 2, _level_size(case, l)), lats[l]) for l in range(3)]
        tr = torch.linalg.inv(_dense(D[2], lat, dof)).diagonal().sum()
        y = [D[1](x[1]), D[2](x[2]), P[0].restrict(x[0]), P[0].prolong(x[1])]
        return [v.reshape(2, -1) for v in y] + [np.array([float(tr.real), float(tr.imag)])]
    # estimate: the samples x^H O_l x and x^H F_l x of every level, and of the coarsest inverse
    D, P, lat, dof = _levels(case, seed, U, 2, 12)
    k, lats = case['samples'], [dims, P[0].nc, P[1].nc]
    dofs = [12, 2 * P[0].ntv, 2 * P[1].ntv]
    inv = [None] + [torch.linalg.inv(_dense(D[l], lats[l], dofs[l])) for l in (1, 2)]

    def solve(l, v):
        if l == 0:
            return _solve(D[0], v)
        return (v.reshape(v.shape[0], -1) @ inv[l].transpose(0, 1)).reshape(v.shape)

    def form(a, b):
        return (a.conj() * b).flatten(1).sum(1)

    def noise(l, term):
        return _field(_z4(_level_size(case, l), seed, 0, term, k), lats[l])

    out = []
    for l in (0, 1):
        x = noise(l, 16 + l)
        y = x - P[l].prolong(P[l].restrict(x))
        out.append(form(y, solve(l, y)))
    for l in (0, 1):
        x = noise(l + 1, 32 + l)
        y = P[l].prolong(x)
        out.append(form(y, solve(l, y)) - form(x, solve(l + 1, x)))
    x = noise(2, 48)
    out.append(form(x, solve(2, x)))
    return out
