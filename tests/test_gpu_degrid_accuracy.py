"""Degridding with the factored kernels is as exact as with the FP32 sums that
they took the place of: items of few visibilities (the FP32 kernel that spreads a
visibility over several lanes) and Stokes I (FP32 sums of XX and YY).  Both
against the FP64 oracle on the same inputs."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_many_kinds import _obs, _same_as_alone

pytestmark = pytest.mark.gpu

# The errors are sums over pixels of independent roundings, so their rms over 1700 or more complex values and four
# observations is known to 1 %; the factored form adds the halves' 2^-23 of either operand and
# what is left of the accumulation's truncation to the one __sincosf that both have: 10 % with both.
MARGIN = 1.10


def _error(idg_mod, oracle_mod, L, n_ch, n_t, steps, stokes, seed):
    import torch
    rng = np.random.default_rng(seed)
    obs = synth.make_observation(synth.stations_uniform_disk(rng, 9, 900.0), n_t, 2.0, np.linspace(140e6, 170e6, n_ch),
                                 steps, 1024, L, 12 if L == 32 else 18, 0.5)
    A = synth.aterms_random(rng, obs.n_intervals, obs.n_stations, obs.aterm_nodes).astype(np.complex64)
    if stokes:
        A[..., 1:3] = 0.0
    geom = oracle_mod.Geometry(obs.grid_size, L, obs.kernel_padding, obs.image_size, aterm_nodes=obs.aterm_nodes,
                               flags=oracle_mod.FLAG_STOKES_I if stokes else 0)
    pl = oracle_mod.plan(geom, obs.uvw, obs.freqs, obs.aterm_offsets)
    out = []
    for mac in (idg_mod.IDG_MAC_DEFAULT, idg_mod.IDG_MAC_FP32):
        plan = idg_mod.Plan(obs, mac_unit=mac, flags=idg_mod.IDG_STOKES_I if stokes else 0)
        try:
            want = idg_mod.IDG_KERNEL_FP32 if mac else idg_mod.IDG_KERNEL_FACTORED
            assert plan.kernels()[1] == want
            if not out:
                shape = plan.grid_shape()
                G = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * 1e-3
                ref = oracle_mod.degrid(geom, obs.n_stations, obs.baselines, obs.uvw, obs.freqs, obs.aterm_offsets, pl, G,
                                        A.astype(np.complex128))
            V = torch.empty((obs.n_baselines, obs.n_timesteps, obs.n_channels, 4), dtype=torch.complex64, device="cuda")
            plan.degrid(torch.as_tensor(G).cuda(), torch.as_tensor(A).cuda(), V)
            plan.synchronize()
            d = V.cpu().numpy() - ref.reshape(tuple(V.shape))
            out.append(np.linalg.norm(d.ravel()) / np.linalg.norm(ref.ravel()))
        finally:
            plan.close()
    return out


@pytest.mark.parametrize("L", [32, 64, 96, 128])
@pytest.mark.parametrize("n_ch,n_t,steps,stokes", [(1, 12, 1, False), (1, 16, 2, False), (2, 12, 2, False), (16, 14, 4, True)])
def test_no_larger_error_than_fp32_sums(idg_mod, oracle_mod, cuda_device, L, n_ch, n_t, steps, stokes):
    e = np.mean([_error(idg_mod, oracle_mod, L, n_ch, n_t, steps, stokes, s) for s in range(4)], axis=0)
    assert e[0] < MARGIN * e[1], e


@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0)])
@pytest.mark.parametrize("L,stokes", [(64, False), (128, False), (128, True)])
def test_plans_of_few_visibilities_share_a_call(idg_mod, cuda_device, L, stokes, order):
    """Plans of segments of 2, of 36 and of 12 visibilities in one call: the first has a launch of its own."""
    sizes = [(1, 16, 2), (9, 16, 4), (1, 24, 12)]
    obs_list = [_obs(L=L, n_ch=c, n_t=t, seed=20 + k) for k, (c, t, _) in enumerate(sizes)]
    for o, (_, t, steps) in zip(obs_list, sizes):
        o.aterm_offsets = np.arange(0, t + 1, steps, dtype=np.int32)
    obs_list = [obs_list[k] for k in order]
    plans = [idg_mod.Plan(o, flags=idg_mod.IDG_STOKES_I if stokes else 0) for o in obs_list]
    try:
        assert all(p.kernels()[1] == idg_mod.IDG_KERNEL_FACTORED for p in plans)
        _same_as_alone(idg_mod, plans, obs_list)
    finally:
        for p in plans:
            p.close()
