"""The kernels of one phasor per visibility and pixel (tensor cores, and FP32
with Stokes I) against the FP64 oracle, on plans that are shown to run them:
stations at very different heights and a wide field leave w ranges that the
factored phasors do not take.  w layers with mirrored rows throughout;
tolerances as elsewhere (1e-5)."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_parity import DEGRID_TOL, GRID_TOL, _degrid_err, _rel

pytestmark = pytest.mark.gpu


def _obs(L, n_ch, n_t, steps, irregular=False):
    rng = np.random.default_rng(L + n_ch)
    enu = synth.stations_uniform_disk(rng, 7, 900.0)
    enu[:, 2] = rng.normal(0.0, 300.0, 7)
    freqs = np.linspace(140e6, 170e6, n_ch)
    if irregular:
        freqs = freqs + np.linspace(0.0, 1.0, n_ch) ** 2 * 2e5
    dt = 2.0 if n_ch > 8 else (60.0 if n_ch > 1 else 200.0)  # few channels: w has to move with time
    return synth.make_observation(enu, n_t, dt, freqs, steps, 1024, L, 12 if L == 32 else 18, 0.8)


def _check(idg_mod, oracle_mod, obs, kernels, mac=0, flags=0, diagonal=None):
    import torch
    rng = np.random.default_rng(obs.n_channels)
    A = synth.aterms_random(rng, obs.n_intervals, obs.n_stations, obs.aterm_nodes).astype(np.complex64)
    if diagonal == "all":
        A[..., 1:3] = 0.0
    elif diagonal == "mixed":
        A[::2, ::2, ..., 1:3] = 0.0
    vis = synth.random_visibilities(rng, obs).astype(np.complex64)
    stokes = flags & idg_mod.IDG_STOKES_I
    geom = oracle_mod.Geometry(obs.grid_size, obs.subgrid_size, obs.kernel_padding, obs.image_size,
                               aterm_nodes=obs.aterm_nodes,
                               flags=oracle_mod.FLAG_W_LAYERS | (oracle_mod.FLAG_STOKES_I if stokes else 0))
    pl = oracle_mod.plan(geom, obs.uvw, obs.freqs, obs.aterm_offsets)
    args = (geom, obs.n_stations, obs.baselines, obs.uvw, obs.freqs, obs.aterm_offsets, pl)
    plan = idg_mod.Plan(obs, flags=flags | idg_mod.IDG_W_LAYERS, mac_unit=mac)
    try:
        assert plan.kernels() == kernels
        assert pl.conj.any() and not pl.conj.all()
        A_d = torch.as_tensor(A).cuda()
        G = torch.zeros(plan.grid_shape(), dtype=torch.complex128, device="cuda")
        plan.grid(torch.as_tensor(vis).cuda(), A_d, G)
        plan.synchronize()
        assert _rel(G.cpu().numpy(), oracle_mod.grid(*args, vis.astype(np.complex128), A.astype(np.complex128))) < GRID_TOL
        Gin = (rng.standard_normal(G.shape) + 1j * rng.standard_normal(G.shape)) * 1e-3
        V = torch.full(vis.shape, 7.0 + 7.0j, dtype=torch.complex64, device="cuda")
        plan.degrid(torch.as_tensor(Gin).cuda(), A_d, V)
        plan.synchronize()
        assert _degrid_err(V.cpu().numpy(), oracle_mod.degrid(*args, Gin, A.astype(np.complex128))) < DEGRID_TOL
    finally:
        plan.close()


@pytest.mark.parametrize("persistent", [False, True])
# row groups and runs of every length, items of one and two segments, few-lane items only (1 and 2 channels)
@pytest.mark.parametrize("n_ch,n_t,steps", [(24, 12, 4), (17, 7, 3), (5, 9, 1), (2, 6, 2), (1, 12, 4)])
@pytest.mark.parametrize("L", [32, 64, 96, 128])
def test_tensor_kernels(idg_mod, oracle_mod, cuda_device, L, n_ch, n_t, steps, persistent):
    T = idg_mod.IDG_KERNEL_TENSOR
    _check(idg_mod, oracle_mod, _obs(L, n_ch, n_t, steps), (T, T), flags=idg_mod.IDG_PERSISTENT if persistent else 0)


@pytest.mark.parametrize("diagonal", [None, "all", "mixed"])
@pytest.mark.parametrize("unit", ["default", "tensor"])
@pytest.mark.parametrize("L", [32, 64, 96, 128])
def test_stokes_i(idg_mod, oracle_mod, cuda_device, L, unit, diagonal):
    """By default on the FP32 kernels, by request on the tensor-core ones."""
    k = idg_mod.IDG_KERNEL_FP32 if unit == "default" else idg_mod.IDG_KERNEL_TENSOR
    _check(idg_mod, oracle_mod, _obs(L, 11, 8, 3), (k, k), flags=idg_mod.IDG_STOKES_I, diagonal=diagonal,
           mac=0 if unit == "default" else idg_mod.IDG_MAC_TENSOR)


@pytest.mark.parametrize("L", [32, 64, 96, 128])
def test_irregular_channels(idg_mod, oracle_mod, cuda_device, L):
    _check(idg_mod, oracle_mod, _obs(L, 13, 8, 3, irregular=True), (idg_mod.IDG_KERNEL_FP32, idg_mod.IDG_KERNEL_TENSOR))
