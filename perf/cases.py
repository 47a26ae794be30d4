"""Measured cases of the library's hot path.

Each case is one call, or one short sequence of calls, that a program using this package makes in earnest: local
energies, log psi, Markov-chain sampling, local derivatives, the vector-Jacobian product behind autograd, and the
stochastic-reconfiguration solve. `listed` names the cases that are followed over time, `draw` gives others from the
same ranges, `prepare` makes what the caller holds before the call, `run` makes the call, `work` counts what the path
cannot do without, and `exact` evaluates the same quantities in float64 with plain torch.

Lattices, networks and batch sizes are those of `nqs_synth.WORKLOADS`, the serving mix and the tests of this
repository.
"""

import math

import numpy as np
import torch

import nqs_synth
from paper_2204_07816_gb300 import autograd, nqs

# dense forward FLOPs that the float64 reference may take before it would need too long
EXACT_FLOPS = 8e12


def _case(kind, model, L, channels, layers, n, prec='bf16', **more):
    d = dict(kind=kind, model=model, L=L, channels=channels, layers=layers, n=n, prec=prec, scale=0.5)
    d.update(more)
    return d


def listed():
    cases = [
        # a short evaluation of the wave function (a minibatch of an outer loop): launches and host time count
        ('logpsi_small', _case('logpsi', 'j1j2', 10, 16, 6, 64)),
        # the parity workload in the default precision: small network, float64, four channels
        ('eloc_4x4_fp64', _case('eloc', 'j1j2', 4, 4, 2, 1024, 'fp64')),
        # the local energies of one step of the 10x10 workload, the call that dominates an optimisation
        ('eloc_10x10', _case('eloc', 'j1j2', 10, 16, 6, 8192)),
        # the largest network of the workloads
        ('eloc_16x16', _case('eloc', 'j1j2', 16, 32, 8, 4096)),
        # the t-J workload: hops, exchanges, three one-hot input channels
        ('eloc_tj_12x12', _case('eloc', 'tj', 12, 32, 6, 2048)),
        # the float32 path on a validation subset of the 10x10 workload
        ('eloc_10x10_fp32', _case('eloc', 'j1j2', 10, 16, 6, 512, 'fp32')),
        # serving: what a batcher has pending from several requests, uneven lattices, both Hamiltonians, two widths
        ('eloc_group', _case('group', 'mixed', 12, 16, 4, 2048)),
        # one step's sampling on the 10x10 workload (256 chains, some sweeps), freshly initialised network
        ('sample_10x10', _case('sample', 'j1j2', 10, 16, 6, 256, sweeps=8)),
        # t-J sampling with a more structured wave function (lower acceptance)
        ('sample_tj_12x12', _case('sample', 'tj', 12, 32, 6, 256, sweeps=2, scale=1.5)),
        # local derivatives of every sample of a step
        ('grad_10x10', _case('grad', 'j1j2', 10, 16, 6, 8192)),
        # a loss differentiated through log psi with torch.autograd, the wide network
        ('vjp_16x16', _case('vjp', 'j1j2', 16, 32, 8, 2048)),
        # the stochastic-reconfiguration solve and update of a 10x10 step
        ('sr_10x10', _case('sr', 'j1j2', 10, 16, 6, 8192, eps=1e-4)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(['logpsi', 'eloc', 'eloc', 'eloc', 'group', 'sample', 'grad', 'vjp', 'sr'])
    model = rng.choice(['j1j2', 'j1j2', 'tj'])
    channels = rng.choice([16, 16, 32])
    L = rng.randint(4, 16)
    layers = rng.randint(2, 8)
    prec = 'bf16'
    if kind in ('eloc', 'logpsi', 'grad') and rng.random() < 0.3:   # the CUDA-core precisions
        prec = rng.choice(['fp32', 'fp32', 'fp64'])
        channels = rng.choice([4, 8, 16])
        L = rng.randint(4, 12)
        layers = rng.randint(2, 6)
    c = _case(kind, model, L, channels, layers, 0, prec)
    if kind == 'eloc' and prec == 'bf16' and channels == 16 and rng.random() < 0.3:
        plan = nqs.tc_plan(_problem(c), 'local_energy', 1024)
        if plan is not None and plan['row_form'] == 1:
            c['prec'] = 'fp8'
    if kind == 'logpsi':
        c['n'] = _log_int(rng, 1, 16384)
    elif kind == 'eloc':
        c['n'] = _log_int(rng, 8, 8192)
    elif kind == 'group':
        c.update(model='mixed', L=rng.randint(6, 14), n=_log_int(rng, 64, 4096))
    elif kind == 'sample':
        c.update(n=_log_int(rng, 16, 1024), sweeps=rng.randint(1, 4), scale=rng.choice([0.5, 1.0, 1.5]))
    elif kind in ('grad', 'vjp'):
        c['n'] = _log_int(rng, 8, 8192)
    else:
        c.update(n=_log_int(rng, 16, 8192), eps=rng.choice([1e-4, 1e-3]), layers=rng.randint(2, 6))
    # keep a drawn case's work below that of the largest listed one (float32 and float64 run on the CUDA cores)
    top = work(dict(listed()[3]))['flops']
    share = {'bf16': 0.5, 'fp8': 0.5, 'fp32': 1 / 60, 'fp64': 1 / 600}[c['prec']]
    if kind in ('grad', 'vjp'):
        share = min(share, 1 / 15 if c['prec'] != 'fp64' else 1 / 2000)
    if kind == 'sample':
        share /= 15
    unit = work(dict(c, n=max(c['n'], 1)))['flops'] / max(c['n'], 1)
    c['n'] = max(1, min(c['n'], int(top * share / unit)))
    if kind in ('grad', 'sr'):   # the [2 n, P] matrix
        c['n'] = max(1, min(c['n'], int(4e9 / (16 * _n_params(c)))))
    return c


# ---------------------------------------------------------------- problems and inputs
def _c_in(c):
    return 1 if c['model'] == 'j1j2' else 3


def _fill(c):
    """(n_up, n_down): half filling for J1-J2, one hole in eight sites for t-J."""
    N = c['L'] ** 2
    electrons = N if c['model'] == 'j1j2' else N - N // 8
    return electrons // 2, electrons - electrons // 2


def _problem(c):
    n_up, n_down = _fill(c)
    return nqs.make_problem(c['model'], c['L'], n_up=n_up, n_down=n_down, n_layers=c['layers'], channels=c['channels'])


def _n_params(c):
    return nqs_synth.n_params(_c_in(c), c['channels'], c['layers'])


def _members(c):
    """The requests of a grouped call: uneven lattices, models and widths around the case's own."""
    L, n = c['L'], c['n']
    shapes = [('j1j2', L, 16, 1), ('j1j2', max(4, L - 4), 16, 2), ('tj', max(4, L - 6), 16, 2), ('j1j2', 6, 16, 4),
              ('tj', L, 32, 4), ('j1j2', max(4, L - 2), 32, 4)]
    return [_case('eloc', m, l, ch, c['layers'], max(1, n // div)) for m, l, ch, div in shapes]


def _params(c, seed):
    return nqs_synth.random_params(_c_in(c), c['channels'], c['layers'], seed + 1, scale=c['scale'])


def _configs(c, seed):
    n_up, n_down = _fill(c)
    return nqs_synth.random_configs(c['L'] ** 2, n_up, n_down, c['n'], seed + 2)


def _context(c, seed):
    p = torch.tensor(_params(c, seed), dtype=torch.float64, device='cuda')
    return nqs.Context(_problem(c), p, seed=seed)


def _sr_inputs(c, seed):
    """O as a step hands it to the solver (the float32 derivatives of its samples, in float64 storage) and local
    energies that correlate with it."""
    params = torch.tensor(_params(c, seed), dtype=torch.float32, device='cuda')
    cfg = torch.from_numpy(_configs(c, seed)).cuda()
    O = torch.empty((2 * c['n'], _n_params(c)), dtype=torch.float64, device='cuda')
    _derivatives(params, cfg, c, O)
    gen = torch.Generator(device='cuda').manual_seed(seed + 3)
    N = c['L'] ** 2
    w = torch.randn(O.shape[1], generator=gen, device='cuda', dtype=torch.float64) * 1e-3
    noise = torch.randn((c['n'], 2), generator=gen, device='cuda', dtype=torch.float64) * (0.02 * math.sqrt(N))
    proj = (O @ w).reshape(2, -1).t()
    e = proj - proj.mean(0) + noise
    e[:, 0] += 0.75 * N
    return O, e.contiguous()


def prepare(case, seed):
    c, kind = case, case['kind']
    if kind == 'group':
        ms = _members(c)
        return dict(kind=kind, prec=c['prec'], ctxs=[_context(m, seed + 10 * i) for i, m in enumerate(ms)],
                    cfgs=[torch.from_numpy(_configs(m, seed + 10 * i)).cuda() for i, m in enumerate(ms)])
    s = dict(kind=kind, prec=c['prec'], ctx=_context(c, seed))
    if kind == 'sr':
        s['O'], s['e'] = _sr_inputs(c, seed)
        s['start'] = s['ctx'].params.clone()
        s['eps'] = c['eps']
        return s
    s['cfg'] = torch.from_numpy(_configs(c, seed)).cuda()
    if kind == 'sample':
        s['sweeps'] = c['sweeps']
    if kind == 'vjp':
        s['ctx'].params.requires_grad_(True)
        gen = torch.Generator().manual_seed(seed + 4)
        s['g'] = torch.randn((c['n'], 2), generator=gen, dtype=torch.float64).cuda() / c['n']
    return s


def run(state):
    s, kind, prec = state, state['kind'], state['prec']
    if kind == 'logpsi':
        return s['ctx'].logpsi(s['cfg'], prec)
    if kind == 'eloc':
        return s['ctx'].local_energy(s['cfg'], None, prec)
    if kind == 'group':
        return nqs.local_energy_multi(s['ctxs'], s['cfgs'], prec)
    if kind == 'sample':   # resumed from the checkpointed chains: one sample a sweep
        s['ctx'].set_chains(s['cfg'], 0)
        cfg, logpsi = s['ctx'].sample(s['cfg'].shape[0], s['sweeps'], 1, 0, prec)
        return {'configs': cfg, 'logpsi': logpsi}
    if kind == 'grad':
        return s['ctx'].logpsi_grad(s['cfg'], prec)
    if kind == 'vjp':
        params = s['ctx'].params
        lp = autograd.logpsi(params, s['cfg'], s['ctx'], prec)
        (grad,) = torch.autograd.grad(lp, params, s['g'])
        return {'logpsi': lp.detach(), 'grad': grad}
    # sr: the solve and the update from the same parameters in every pass
    s['ctx'].params.copy_(s['start'])
    delta, _ = s['ctx'].sr_solve(s['O'], s['e'], eps=s['eps'], rtol=1e-8, lr=0.02, apply_update=True)
    return {'delta': delta, 'params': s['ctx'].params}


# ---------------------------------------------------------------- work
def _layer_flops(c, l):
    return 2.0 * 9 * (_c_in(c) if l == 0 else c['channels']) * c['channels']


def _dense_flops(c):
    return c['L'] ** 2 * sum(_layer_flops(c, l) for l in range(c['layers']))


def _cone_flops(c, diagonal):
    """One forward restricted to the sites whose activations change when a bond's two sites are exchanged."""
    N, f = c['L'] ** 2, 0.0
    for l in range(c['layers']):
        r = l + 1
        sites = (2 * r + 1) ** 2 + (4 * r + 1 if diagonal else 2 * r + 1)
        f += _layer_flops(c, l) * min(N, sites)
    return f


def _changing(c):
    """Expected fraction of bonds whose two sites differ."""
    n_up, n_down = _fill(c)
    N = c['L'] ** 2
    holes = N - n_up - n_down
    return 1.0 - sum(k * (k - 1) for k in (n_up, n_down, holes)) / (N * (N - 1.0))


def work(case):
    c, kind = case, case['kind']
    if kind == 'group':
        parts = [work(m) for m in _members(c)]
        return {k: sum(p[k] for p in parts) for k in ('bytes', 'flops')}
    n, N, P = c['n'], c['L'] ** 2, _n_params(c)
    if kind == 'logpsi':
        return {'bytes': n * (N + 16) + 8 * P, 'flops': n * _dense_flops(c)}
    if kind == 'eloc':
        conn = _changing(c) * 2 * N * _cone_flops(c, False)
        if c['model'] == 'j1j2':
            conn += _changing(c) * 2 * N * _cone_flops(c, True)
        return {'bytes': n * (N + 16) + 8 * P, 'flops': n * (_dense_flops(c) + conn)}
    if kind == 'sample':
        moves = n * c['sweeps'] * N * _changing(c)
        return {'bytes': n * N + n * c['sweeps'] * (N + 16) + 8 * P, 'flops': moves * _cone_flops(c, False)}
    if kind in ('grad', 'vjp'):
        # forward, then per output stream the weight gradient and the gradient of every layer input but the first
        streams = 2 if kind == 'grad' else 1
        fwd = _dense_flops(c)
        back = streams * (2 * fwd - N * _layer_flops(c, 0))
        out = 16 * n * P if kind == 'grad' else 32 * n + 8 * P
        return {'bytes': n * N + 8 * P + out, 'flops': n * (fwd + back)}
    # sr: O and the energies once, the update; one application of S
    return {'bytes': 16 * n * P + 16 * n + 24 * P, 'flops': 8.0 * n * P}


# ---------------------------------------------------------------- float64 reference in plain torch
def _neighbours(L):
    s = torch.arange(L * L)
    x, y = s % L, s // L
    return torch.stack([((y + dy) % L) * L + (x + dx) % L for dy in (-1, 0, 1) for dx in (-1, 0, 1)])


def _unpack(params, c):
    layers, off, C = [], 0, c['channels']
    for l in range(c['layers']):
        ci = _c_in(c) if l == 0 else C
        W = params[off:off + 9 * ci * C].reshape(C, ci, 9)
        off += 9 * ci * C
        layers.append((W, params[off:off + C]))
        off += C
    return layers, params[off:off + C], params[off + C:off + 2 * C]


def _encode(cfg, c, dtype):
    if c['model'] == 'j1j2':
        return cfg.to(dtype)[:, :, None]
    return torch.stack([cfg == 0, cfg == 1, cfg == -1], dim=2).to(dtype)


def _columns(h, nbr):
    B, N, C = h.shape
    return h[:, nbr.t().reshape(-1), :].reshape(B, N, 9 * C)


def _forward(params, cfg, c, keep=False):
    layers, wa, wp = _unpack(params, c)
    nbr = _neighbours(c['L']).to(cfg.device)
    h, kept = _encode(cfg, c, params.dtype), []
    for W, b in layers:
        cols = _columns(h, nbr)
        z = cols @ W.permute(2, 1, 0).reshape(-1, W.shape[0]) + b
        h = z * torch.sigmoid(z)
        if keep:
            kept.append((cols, z))
    hbar = h.sum(1)
    out = torch.stack([hbar @ wa, hbar @ wp], dim=1)
    return (out, hbar, kept) if keep else out


def _chunks(n, per_item, budget=4e9):
    step = max(1, int(budget / per_item))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _forward_all(params, cfg, c):
    per = 9 * c['channels'] * c['L'] ** 2 * 8 * 3
    return torch.cat([_forward(params, cfg[a:b], c) for a, b in _chunks(cfg.shape[0], per)])


def _derivatives(params, cfg, c, O):
    """Rows d a / d theta, then d phi / d theta, of every configuration into O [2 n, P]."""
    layers, wa, wp = _unpack(params, c)
    nbr = _neighbours(c['L']).to(cfg.device)
    back = nbr.flip(0)   # the site at -d
    n, C, N = cfg.shape[0], c['channels'], c['L'] ** 2
    per = (9 * C * N * (c['layers'] + 4) + 4 * params.numel()) * params.element_size()
    for a, b in _chunks(n, per):
        _, hbar, kept = _forward(params, cfg[a:b], c, keep=True)
        for stream, w in ((0, wa), (1, wp)):
            rows = torch.zeros((b - a, params.numel()), dtype=params.dtype, device=cfg.device)
            end = params.numel() - 2 * C
            rows[:, end + stream * C:end + (stream + 1) * C] = hbar
            g = w.expand(b - a, N, C)
            for l in range(c['layers'] - 1, -1, -1):
                W = layers[l][0]
                cols, z = kept[l]
                s = torch.sigmoid(z)
                gz = g * (s * (1 + z * (1 - s)))
                ci = W.shape[1]
                rows[:, end - C:end] = gz.sum(1)
                dW = torch.bmm(cols.transpose(1, 2), gz).reshape(b - a, 9, ci, C).permute(0, 3, 2, 1)
                rows[:, end - C - 9 * ci * C:end - C] = dW.reshape(b - a, -1)
                end -= C + 9 * ci * C
                if l > 0:
                    g = _columns(gz, back) @ W.permute(2, 0, 1).reshape(-1, ci)
            O[stream * n + a:stream * n + b] = rows.to(O.dtype)


def _bonds(c):
    L = c['L']
    s = torch.arange(L * L)
    x, y = s % L, s // L
    out = []
    for d, (dx, dy) in enumerate([(1, 0), (0, 1), (1, 1), (1, -1)][:4 if c['model'] == 'j1j2' else 2]):
        j = ((y + dy) % L) * L + (x + dx) % L
        out += [(int(a), int(b), d >= 2) for a, b in zip(s, j)]
    return out


def _local_energy(params, cfg, c):
    """H_SS + sum over the bonds that change S of <S|H|S'> W(S') / W(S), couplings J1 = 1, J2 = 0.5 or t = 1, J = 0.4."""
    n, L = cfg.shape[0], c['L']
    v = cfg.to(torch.float64)
    base = _forward_all(params, cfg, c)
    diag = torch.zeros(n, dtype=torch.float64, device=cfg.device)
    off = torch.zeros(n, dtype=torch.complex128, device=cfg.device)
    if c['model'] == 'tj':
        site = torch.arange(L * L)
        x, y = site % L, site // L
        pos = y * L + torch.where(y % 2 == 0, x, L - 1 - x)
        order = torch.argsort(pos)
        occ = (cfg[:, order.to(cfg.device)] != 0).to(torch.int64)
        cum = torch.cat([torch.zeros((n, 1), dtype=torch.int64, device=cfg.device), occ.cumsum(1)], 1)
    pend_cfg, pend_row, pend_h, held = [], [], [], 0

    def flush():
        if not pend_cfg:
            return
        row, h = torch.cat(pend_row), torch.cat(pend_h)
        lp = _forward_all(params, torch.cat(pend_cfg), c) - base[row]
        term = h * torch.exp(lp[:, 0]) * torch.exp(1j * lp[:, 1])
        off.index_add_(0, row, term)
        pend_cfg.clear(), pend_row.clear(), pend_h.clear()

    for i, j, nnn in _bonds(c):
        si, sj = v[:, i], v[:, j]
        if c['model'] == 'j1j2':
            Jb = 0.5 if nnn else 1.0
            diag += 0.25 * Jb * si * sj
            h = torch.where(si != sj, 0.5 * Jb, 0.0)
        else:
            both = (si != 0) & (sj != 0)
            diag += torch.where(both, 0.4 * (0.25 * si * sj - 0.25), 0.0)
            lo, hi = sorted((int(pos[i]), int(pos[j])))
            sign = 1.0 - 2.0 * ((cum[:, hi] - cum[:, lo + 1]) % 2)
            h = torch.where(both & (si != sj), 0.2, torch.where((si == 0) != (sj == 0), -1.0 * sign, 0.0))
        row = torch.nonzero(h).flatten()
        if row.numel() == 0:
            continue
        s2 = cfg[row].clone()
        s2[:, i], s2[:, j] = cfg[row, j], cfg[row, i]
        pend_cfg.append(s2), pend_row.append(row), pend_h.append(h[row].to(torch.float64))
        held += row.numel()
        if held >= 1 << 17:
            flush()
            held = 0
    flush()
    return torch.stack([diag + off.real, off.imag], dim=1)


def _sr_solution(O, e, eps, P):
    """(S + eps I) delta = F by conjugate gradient in float64, run to the arithmetic's limit."""
    n = e.shape[0]
    means = torch.stack([O[:n].mean(0), O[n:].mean(0)])
    eh = (e - e.mean(0)).t().reshape(-1)

    def apply(v):
        y = O @ v
        y[:n] -= means[0] @ v
        y[n:] -= means[1] @ v
        return (O.t() @ y - means[0] * y[:n].sum() - means[1] * y[n:].sum()) / n + eps * v

    F = (O.t() @ eh - means[0] * eh[:n].sum() - means[1] * eh[n:].sum()) / n
    x, r = torch.zeros_like(F), F.clone()
    p, rs = r.clone(), r @ r
    stop = float(rs) * 1e-28
    for _ in range(2000):
        if float(rs) <= stop:
            break
        Ap = apply(p)
        alpha = rs / (p @ Ap)
        x += alpha * p
        r -= alpha * Ap
        new = r @ r
        p = r + (new / rs) * p
        rs = new
    return x


def _exact_flops(c):
    if c['kind'] == 'group':
        return sum(_exact_flops(m) for m in _members(c))
    bonds = _changing(c) * (4 if c['model'] == 'j1j2' else 2) * c['L'] ** 2
    return c['n'] * _dense_flops(c) * ((1 + bonds) if c['kind'] == 'eloc' else 5)


def exact(case, seed):
    c, kind = case, case['kind']
    if kind == 'sample' or _exact_flops(c) > EXACT_FLOPS:
        return None   # the chains' states are whole numbers, and log psi follows them
    if kind == 'group':
        return [exact(m, seed + 10 * i) for i, m in enumerate(_members(c))]
    params = torch.tensor(_params(c, seed), dtype=torch.float64, device='cuda')
    if kind == 'sr':
        O, e = _sr_inputs(c, seed)
        delta = _sr_solution(O, e, c['eps'], params.numel())
        return {'delta': delta, 'params': params - 0.02 * delta}
    cfg = torch.from_numpy(_configs(c, seed)).cuda()
    if kind == 'logpsi':
        return _forward_all(params, cfg, c)
    if kind == 'eloc':
        return _local_energy(params, cfg, c)
    O = torch.empty((2 * c['n'], params.numel()), dtype=torch.float64, device='cuda')
    if kind == 'grad':
        _derivatives(params, cfg, c, O)
        return O
    gen = torch.Generator().manual_seed(seed + 4)
    g = torch.randn((c['n'], 2), generator=gen, dtype=torch.float64).cuda() / c['n']
    _derivatives(params, cfg, c, O)
    return {'logpsi': _forward_all(params, cfg, c), 'grad': g.t().reshape(-1) @ O}
