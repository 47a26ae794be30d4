"""Grouped local energies across problems (nqs_local_energy_multi) and the
chunked bond enumeration of large lattices, against the single-problem
entry point and the FP64 oracle."""

import numpy as np
import pytest
import torch

import nqs_synth
from oracle import eloc
from tests.gpu_common import WL, configs_for, dev, lib, make_ctx, oracle_of, problem_of

pytestmark = pytest.mark.gpu

MIX = [
    ('j1j2_10x10', {}),
    ('j1j2_10x10', {'L': 6, 'n_up': 18, 'n_down': 18, 'J2': 0.4, 'n_layers': 4}),
    ('tj_12x12', {'L': 6, 'n_up': 15, 'n_down': 14, 'channels': 16, 'n_layers': 3}),
    ('j1j2_16x16', {'n_layers': 3}),
    ('tj_12x12', {}),
    ('j1j2_10x10', {'L': 8, 'n_up': 32, 'n_down': 32, 'channels': 32, 'n_layers': 3}),
]


@pytest.mark.parametrize('prec', ['bf16', 'fp64'])
def test_grouped_equals_single_problem_launches(prec):
    nqs = lib()
    mix = MIX if prec == 'bf16' else MIX[:3]
    ctxs, cfgs, singles = [], [], []
    for i, (name, over) in enumerate(mix):
        w = WL[name]
        ctx, _ = make_ctx(w, param_seed=10 + i, **over)
        cfg = dev(configs_for(w, 5 + 3 * i, seed=20 + i, **over))
        ctxs.append(ctx)
        cfgs.append(cfg)
        singles.append(ctx.local_energy(cfg, None, prec))
    outs = nqs.local_energy_multi(ctxs, cfgs, prec)
    torch.cuda.synchronize()
    for a, b in zip(outs, singles):
        assert torch.equal(a, b)


@pytest.mark.parametrize('count', [22, 24, 33])
def test_grouped_many_requests(count):
    """More requests than one launch of the wide form holds, with members of
    the tap form between them: bitwise the single-problem launches."""
    nqs = lib()
    w = WL['j1j2_10x10']
    kinds = [{'L': 6, 'n_up': 18, 'n_down': 18, 'channels': 32, 'n_layers': 2},
             {'L': 8, 'n_up': 32, 'n_down': 32, 'channels': 32, 'n_layers': 2},
             {'L': 4, 'n_up': 8, 'n_down': 8, 'channels': 32, 'n_layers': 2}]
    ctxs = [make_ctx(w, param_seed=50 + i, **kinds[i % 7 % 3])[0] for i in range(count)]
    cfgs = [dev(configs_for(w, 1 + i % 4, seed=60 + i, **kinds[i % 7 % 3])) for i in range(count)]
    outs = nqs.local_energy_multi(ctxs, cfgs, 'bf16')
    torch.cuda.synchronize()
    for ctx, cfg, got in zip(ctxs, cfgs, outs):
        assert torch.equal(got, ctx.local_energy(cfg, None, 'bf16'))


def test_grouped_rejects_unsupported_channel_count():
    nqs = lib()
    w = WL['j1j2_4x4']
    ctx, _ = make_ctx(w)          # 4 channels
    with pytest.raises(nqs.NQSError) as ei:
        nqs.local_energy_multi([ctx], [dev(configs_for(w, 2, 1))], 'bf16')
    assert ei.value.code == -7


def test_chunked_enumeration_large_lattice_vs_oracle():
    """20 x 20 J1-J2 has 1,600 bonds: the tensor-core E_loc walks them in two
    chunks; energy per site within 1e-4 of the oracle on the same samples."""
    w = WL['j1j2_10x10']
    over = {'L': 20, 'n_up': 200, 'n_down': 200, 'channels': 16, 'n_layers': 2}
    ctx, params = make_ctx(w, **over)
    spec, ham = oracle_of(w, **over)
    cfg = configs_for(w, 2, seed=30, **over)
    got = ctx.local_energy(dev(cfg), None, 'bf16').cpu().numpy()
    want = eloc.local_energy(params, cfg, spec, ham)
    assert abs(got[:, 0].mean() - want.real.mean()) / 400 <= 1e-4
    assert np.abs(got[:, 1] - want.imag).max() / 400 <= 1e-4


def test_chunked_enumeration_36x36_zero_network():
    """36 x 36 (5,184 bonds, six chunks): a zero network gives exactly
    (J1 + J2) N / 2 for every configuration."""
    w = WL['j1j2_10x10']
    over = {'L': 36, 'n_up': 648, 'n_down': 648, 'channels': 16, 'n_layers': 3}
    P = lib().nqs_param_count(problem_of(w, **over))
    ctx, _ = make_ctx(w, params=np.zeros(P), **over)
    e = ctx.local_energy(dev(configs_for(w, 3, seed=31, **over)), None, 'bf16').cpu().numpy()
    assert np.all(e[:, 0] == 0.75 * 1296) and np.all(e[:, 1] == 0.0)


def _grouped(shapes, w='j1j2_10x10', cap=0):
    """(contexts, configurations, grouped energies, launches of the grouped call) of requests (overrides, samples)."""
    nqs = lib()
    ctxs = [make_ctx(WL[w], param_seed=70 + i, **over)[0] for i, (over, _) in enumerate(shapes)]
    cfgs = [dev(configs_for(WL[w], n, seed=80 + i, **over)) for i, (over, n) in enumerate(shapes)]
    before = ctxs[0].kernel_launches()
    outs = nqs.local_energy_multi(ctxs, cfgs, 'bf16', max_blocks=cap)
    return ctxs, cfgs, outs, ctxs[0].kernel_launches() - before


def _square(L, channels, layers):
    return {'L': L, 'n_up': L * L // 2, 'n_down': L * L - L * L // 2, 'channels': channels, 'n_layers': layers}


GROUPS = {
    # one launch holds them all (beside one packing launch a request)
    'many': ([(_square(6 + 2 * (i % 2), 32, 2), 1 + i % 4) for i in range(33)], 1),
    'most': ([(_square(6, 16, 4), 1) for i in range(220)], 1),
    'one more': ([(_square(6, 16, 4), 1) for i in range(221)], 2),
    # more plans than a launch holds
    'plans': ([(_square(L, 32, nl), 2) for nl in (1, 2, 3) for L in (6, 7, 8, 9, 10, 11, 12, 13, 14)], 2),
    # some requests in the tap form only: everything in the tap form, if that is shorter than two launches
    'beside longer': ([(_square(10, 16, 4), 3), (_square(16, 16, 4), 2)], 1),
    'beside shorter': ([(_square(8, 32, 4), 3), (_square(4, 32, 4), 2)], 2),
    'many samples': ([(_square(8, 16, 4), 6000), (_square(16, 16, 2), 2)], 2),
    'more than SMs': ([(_square(10, 16, 4), 150), (_square(16, 16, 4), 20)], 1),
}


@pytest.mark.parametrize('name', list(GROUPS))
def test_grouped_launches(name):
    """How many launches a grouped call takes (requests, plans and forms a launch holds), and bitwise the
    single-problem launches, whichever form a request runs in."""
    shapes, launches = GROUPS[name]
    ctxs, cfgs, outs, count = _grouped(shapes)
    torch.cuda.synchronize()
    assert count == len(shapes) + launches
    for ctx, cfg, got in zip(ctxs, cfgs, outs):
        assert torch.equal(got, ctx.local_energy(cfg, None, 'bf16'))


def test_grouped_cap_is_a_share_of_the_sms():
    """max_blocks counts SMs, also for the form whose blocks take half an SM each: capped at every SM a call is no
    slower than uncapped (1.6 times where it gets half the blocks), and a cap changes no bit."""
    nqs = lib()
    shapes = [(_square(10, 16, 4), 512), (_square(8, 16, 4), 512), (_square(6, 16, 4), 512)]
    ctxs, cfgs, outs, _ = _grouped(shapes)
    for cap in (1, 31):
        few = [c[:40].contiguous() for c in cfgs]
        for a, b in zip(nqs.local_energy_multi(ctxs, few, 'bf16', max_blocks=cap), outs):
            assert torch.equal(a, b[:40])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    best = {}
    for cap in (0, sms) * 4:
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        nqs.local_energy_multi(ctxs, cfgs, 'bf16', outs=outs, max_blocks=cap)
        a.record()
        for _ in range(5):
            nqs.local_energy_multi(ctxs, cfgs, 'bf16', outs=outs, max_blocks=cap)
        b.record()
        torch.cuda.synchronize()
        best[cap] = min(best.get(cap, 1e9), a.elapsed_time(b))
    assert best[sms] <= 1.15 * best[0]
