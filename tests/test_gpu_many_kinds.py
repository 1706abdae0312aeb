"""grid_many / degrid_many over plans whose kernels differ: whether the
phasors can be factored follows from each plan's own w range, so plans of one
geometry may run different kernels and still share a call."""
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
