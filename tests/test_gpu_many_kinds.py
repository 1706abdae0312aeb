"""grid_many / degrid_many over plans whose kernels differ: whether the
phasors can be factored follows from each plan's own w range, so plans of one
geometry may run different kernels and still share a call."""
import itertools

import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_parity import _random_problem

pytestmark = pytest.mark.gpu


def _obs(L=64, fov=0.5, n_ch=9, n_t=8, heights=0.0, n_st=7, seed=1, N=2048):
    """Heights spread |w| over several w layers and widen the w range of every subgrid."""
    rng = np.random.default_rng(seed)
    enu = synth.stations_uniform_disk(rng, n_st, 900.0)
    enu[:, 2] = rng.normal(0.0, heights, n_st) if heights else 0.0
    return synth.make_observation(enu, n_t, 2.0, np.linspace(140e6, 170e6, n_ch), 4, N, L, 18, fov)


def _inputs(plans, obs_list):
    import torch
    A, V, G = [], [], []
    for s, (p, obs) in enumerate(zip(plans, obs_list)):
        a, v = _random_problem(40 + s, obs)
        A.append(torch.as_tensor(a).cuda())
        V.append(torch.as_tensor(v).cuda())
        G.append(torch.zeros(p.grid_shape(), dtype=torch.complex128, device="cuda"))
    return A, V, G


def _timed(fn, n=5):
    import torch
    best = 1e9
    for _ in range(n):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def test_order_of_plans_does_not_size_the_launch(idg_mod, cuda_device):
    """A flat user taper leaves no w range for factored phasors, so the first plan runs the general kernels; the
    factored ones behind it still get a block per SM.  Sized by a plan that knows no SM count they got one block
    per 512 items, 26 times slower here; the order costs nothing else, so a factor of 3 is far from noise."""
    flat = _obs(heights=20.0, n_st=4)
    many = _obs(n_ch=24, n_t=40, n_st=40, seed=2)
    plans = [idg_mod.Plan(flat, taper_user=np.ones(64), flags=idg_mod.IDG_W_LAYERS, mac_unit=idg_mod.IDG_MAC_TENSOR),
             idg_mod.Plan(many, flags=idg_mod.IDG_W_LAYERS, mac_unit=idg_mod.IDG_MAC_TENSOR)]
    try:
        A, V, G = _inputs(plans, [flat, many])
        rev = [x[::-1] for x in (plans, V, A, G)]
        idg_mod.grid_many(plans, V, A, G)
        idg_mod.degrid_many(plans, G, A, V)
        for call, args, back in ((idg_mod.grid_many, (plans, V, A, G), rev),
                                 (idg_mod.degrid_many, (plans, G, A, V), (rev[0], rev[3], rev[2], rev[1]))):
            assert _timed(lambda: call(*args)) < 3 * _timed(lambda: call(*back))
    finally:
        for p in plans:
            p.close()


def _same_as_alone(idg_mod, plans, obs_list, stokes_i=False):
    import torch
    A, V, G = _inputs(plans, obs_list)
    idg_mod.grid_many(plans, V, A, G)
    outs = [torch.full_like(v, 7.0 + 7.0j) for v in V]
    idg_mod.degrid_many(plans, G, A, outs)
    torch.cuda.synchronize()
    for p, v, a, g, o in zip(plans, V, A, G, outs):
        ref, out = torch.zeros_like(g), torch.full_like(v, 7.0 + 7.0j)
        p.grid(v, a, ref)
        p.degrid(g, a, out)
        p.synchronize()
        # the same kernels: only the order of FP64 and of shared-memory additions differs
        assert float(torch.linalg.vector_norm(g - ref) / torch.linalg.vector_norm(ref)) < 1e-12
        assert float((o - out).abs().max() / out.abs().max()) < 1e-6


FACTORED, GENERAL = dict(), dict(fov=0.8, heights=300.0)


@pytest.mark.parametrize("order", [(0, 1, 0), (1, 0, 1)])
@pytest.mark.parametrize("L", [32, 64, 96, 128])
@pytest.mark.parametrize("kind", ["tensor", "stokes", "irregular"])
def test_plans_of_one_geometry_share_a_call(idg_mod, cuda_device, L, kind, order):
    """Plans inside and outside the bound of the factored phasors, in both orders: four correlations (the tensor-core
    kernels beside the factored ones), Stokes I (the FP32 kernels) and irregularly spaced channels (the FP32 gridder
    and the tensor-core degridder)."""
    F, T, P = idg_mod.IDG_KERNEL_FACTORED, idg_mod.IDG_KERNEL_TENSOR, idg_mod.IDG_KERNEL_FP32
    general = {"tensor": (T, T), "stokes": (P, P), "irregular": (P, T)}[kind]
    obs_list, plans = [], []
    try:
        for s, k in enumerate(order):
            obs = _obs(L=L, seed=5 + s, n_ch=7 + s, N=4096, **(GENERAL if k else FACTORED))
            if L == 32:
                obs.kernel_padding = 12
            if kind == "irregular":
                obs.freqs = obs.freqs + np.linspace(0.0, 1.0, obs.n_channels) ** 2 * 2e5
            obs_list.append(obs)
            plans.append(idg_mod.Plan(obs, flags=idg_mod.IDG_W_LAYERS | (idg_mod.IDG_STOKES_I if kind == "stokes" else 0)))
            assert plans[-1].kernels() == (general if k else (F, F))
        _same_as_alone(idg_mod, plans, obs_list)
    finally:
        for p in plans:
            p.close()


def test_uniform_and_irregular_channels_share_a_call(idg_mod, cuda_device):
    """Both run the factored kernels and report one unit."""
    obs_list = [_obs(seed=9), _obs(seed=10)]
    obs_list[1].freqs = obs_list[1].freqs + np.linspace(0.0, 1.0, obs_list[1].n_channels) ** 2 * 2e5
    plans = [idg_mod.Plan(o) for o in obs_list]
    try:
        assert plans[0].kernels() == plans[1].kernels() and plans[0].stats().mac_unit == plans[1].stats().mac_unit
        _same_as_alone(idg_mod, plans, obs_list)
    finally:
        for p in plans:
            p.close()


def test_answer_does_not_depend_on_the_order(idg_mod, cuda_device):
    """Plans of uniform channels, of irregular ones inside the bound of the factored phasors and of irregular ones
    outside share neither the unit in use nor the one without factored phasors, though each neighbour of the second
    shares one with it: refused in every order.  Any two with the second in common are taken in both."""
    obs_list = [_obs(seed=9), _obs(seed=10), _obs(seed=11, N=4096, **GENERAL)]
    for o in obs_list[1:]:
        o.freqs = o.freqs + np.linspace(0.0, 1.0, o.n_channels) ** 2 * 2e5
    plans = [idg_mod.Plan(o, flags=idg_mod.IDG_W_LAYERS) for o in obs_list]
    try:
        F, T, P = idg_mod.IDG_KERNEL_FACTORED, idg_mod.IDG_KERNEL_TENSOR, idg_mod.IDG_KERNEL_FP32
        assert [p.kernels() for p in plans] == [(F, F), (F, F), (P, T)]
        A, V, G = _inputs(plans, obs_list)
        for n in (2, 3):
            for order in itertools.permutations(range(3), n):
                p, v, a, g = ([x[k] for k in order] for x in (plans, V, A, G))
                for call, args in ((idg_mod.grid_many, (p, v, a, g)), (idg_mod.degrid_many, (p, g, a, v))):
                    if n == 2 and 1 in order:
                        call(*args)
                    else:
                        with pytest.raises(idg_mod.IdgError) as e:
                            call(*args)
                        assert e.value.status == 1
    finally:
        for p in plans:
            p.close()


def test_other_units_are_still_refused(idg_mod, cuda_device):
    obs = _obs(seed=9)
    plans = [idg_mod.Plan(obs, mac_unit=m) for m in (idg_mod.IDG_MAC_TENSOR, idg_mod.IDG_MAC_FP32)]
    try:
        A, V, G = _inputs(plans, [obs, obs])
        for call, args in ((idg_mod.grid_many, (plans, V, A, G)), (idg_mod.degrid_many, (plans, G, A, V))):
            with pytest.raises(idg_mod.IdgError) as e:
                call(*args)
            assert e.value.status == 1
    finally:
        for p in plans:
            p.close()
