"""The separable-phasor kernels (tensor-core plans whose subgrids admit the
separable form of the phase) against the FP64 oracle where their tiles, rings
and scaling can go wrong, and the rule that chooses them: plans outside its
bound keep the general kernels.

Tolerances as elsewhere (1e-5): the split operands and FP32 sums of these
kernels stay near 1e-6, and the neglected terms below 3e-7."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_parity import DEGRID_TOL, GRID_TOL, Case, _degrid_err, _random_problem, _rel

pytestmark = pytest.mark.gpu


def _obs(L, n_ch, n_t, steps, fov=0.5, heights=0.0, nodes=9, n_st=7, N=2048, diameter=900.0):
    rng = np.random.default_rng(n_ch + n_t)
    enu = synth.stations_uniform_disk(rng, n_st, diameter)
    enu[:, 2] = rng.normal(0.0, heights, n_st) if heights else 0.0
    return synth.make_observation(enu, n_t, 2.0, np.linspace(140e6, 170e6, n_ch), steps, N, L, 18 if L > 32 else 12,
                                  fov, aterm_nodes=nodes)


def _check(c, seed):
    assert _rel(c.gpu_grid(), c.oracle_grid()) < GRID_TOL
    rng = np.random.default_rng(seed)
    N = c.obs.grid_size
    Gin = (rng.standard_normal((4, N, N)) + 1j * rng.standard_normal((4, N, N))) * 1e-3
    assert _degrid_err(c.gpu_degrid(Gin), c.oracle_degrid(Gin)) < DEGRID_TOL


# segments of 1, 15, 16, 17 and several hundred visibilities (chunks of 16, rings of 2 to 4 chunks,
# items of at most 64 visibilities), the largest A-term tables
@pytest.mark.parametrize("L,n_ch,n_t,steps,nodes", [(32, 1, 3, 1, 2), (64, 5, 6, 3, 9), (96, 4, 8, 4, 25),
                                                    (128, 17, 4, 1, 25), (64, 31, 20, 20, 9), (32, 33, 9, 5, 25),
                                                    (96, 43, 7, 7, 9), (128, 3, 50, 43, 9)])
def test_separable_segment_sizes(idg_mod, oracle_mod, cuda_device, L, n_ch, n_t, steps, nodes):
    obs = _obs(L, n_ch, n_t, steps, nodes=nodes)
    A, vis = _random_problem(L + n_ch, obs)
    c = Case(idg_mod, oracle_mod, obs, A, vis, mac_unit=idg_mod.IDG_MAC_TENSOR)
    assert c.plan.stats().mac_unit == idg_mod.IDG_MAC_TENSOR
    _check(c, L)


@pytest.mark.parametrize("fov", [0.2, 0.8, 1.2])
def test_wide_fields_keep_the_general_kernels(idg_mod, oracle_mod, cuda_device, fov):
    """At the widest fields n' is no longer separable to the tolerance; either way the results hold."""
    obs = _obs(96, 9, 8, 4, fov=fov, diameter=300.0)
    A, vis = _random_problem(77, obs)
    _check(Case(idg_mod, oracle_mod, obs, A, vis), 5)


def test_values_over_a_wide_range(idg_mod, oracle_mod, cuda_device):
    """Each segment has its own power-of-two scale: baselines of 1e-25, 1e-12, 1e4 and 1e15 times unit
    values, zeros, and an outlier inside a segment; every baseline is checked on its own."""
    import torch
    obs = _obs(64, 6, 8, 4, n_st=5)
    A, vis = _random_problem(3, obs)
    amp = np.array([1e-25, 1e-12, 1e4, 1e15, 1.0, 0.0, 1.0, 1.0, 1e15, 1e-12])
    vis = (vis * amp[:, None, None, None]).astype(np.complex64)
    vis[4, 2, 3] *= 1e5
    c = Case(idg_mod, oracle_mod, obs, A, vis, mac_unit=idg_mod.IDG_MAC_TENSOR)
    for b in range(obs.n_baselines):
        one = np.zeros_like(vis)
        one[b] = vis[b]
        G = torch.zeros((4, obs.grid_size, obs.grid_size), dtype=torch.complex128, device="cuda")
        c.plan.grid(torch.as_tensor(one).cuda(), torch.as_tensor(A).cuda(), G)
        c.plan.synchronize()
        c.vis = one
        ref = c.oracle_grid()
        if amp[b] == 0.0:
            assert not G.any()
        else:
            assert _rel(G.cpu().numpy(), ref) < GRID_TOL


def test_non_finite_values_stay_in_their_subgrids(idg_mod, cuda_device):
    """A NaN or an infinity reaches the cells of the subgrids that hold it and no others."""
    import torch
    obs = _obs(64, 6, 8, 4, n_st=5)
    A, vis = _random_problem(4, obs)
    clean = idg_mod.Plan(obs, mac_unit=idg_mod.IDG_MAC_TENSOR)
    ref = idg_mod.Plan(obs, mac_unit=idg_mod.IDG_MAC_FP32)
    try:
        for bad in (np.nan, np.inf):
            v = vis.copy()
            v[3, 2, 1, 0] = bad
            masks = []
            for p in (clean, ref):
                G = torch.zeros((4, obs.grid_size, obs.grid_size), dtype=torch.complex128, device="cuda")
                p.grid(torch.as_tensor(v).cuda(), torch.as_tensor(A).cuda(), G)
                p.synchronize()
                masks.append(torch.isfinite(torch.view_as_real(G)).all(-1))
            assert not masks[0].all() and torch.equal(masks[0].all(0), masks[1].all(0))
    finally:
        clean.close()
        ref.close()


def test_flat_user_taper_and_layers(idg_mod, oracle_mod, cuda_device):
    """Without a taper the neglected terms count over the whole subgrid (the rule weighs them with it)."""
    obs = _obs(64, 9, 8, 4)
    A, vis = _random_problem(9, obs)
    import torch
    t = np.ones(64)
    geom = oracle_mod.Geometry(obs.grid_size, 64, obs.kernel_padding, obs.image_size, taper_kind=1, taper_user=t)
    pl = oracle_mod.plan(geom, obs.uvw, obs.freqs, obs.aterm_offsets)
    args = (geom, obs.n_stations, obs.baselines, obs.uvw, obs.freqs, obs.aterm_offsets, pl)
    plan = idg_mod.Plan(obs, taper_user=t)
    try:
        G = torch.zeros((4, obs.grid_size, obs.grid_size), dtype=torch.complex128, device="cuda")
        plan.grid(torch.as_tensor(vis).cuda(), torch.as_tensor(A).cuda(), G)
        plan.synchronize()
        G_ref = oracle_mod.grid(*args, vis.astype(np.complex128), A.astype(np.complex128))
        assert _rel(G.cpu().numpy(), G_ref) < GRID_TOL
        V = torch.zeros(vis.shape, dtype=torch.complex64, device="cuda")
        plan.degrid(torch.as_tensor(G_ref).cuda(), torch.as_tensor(A).cuda(), V)
        plan.synchronize()
        assert _degrid_err(V.cpu().numpy(), oracle_mod.degrid(*args, G_ref, A.astype(np.complex128))) < DEGRID_TOL
    finally:
        plan.close()


def test_shared_launch_of_both_kinds(idg_mod, cuda_device):
    """grid_many and degrid_many over plans with and without the separable form."""
    import torch
    obs_list = [_obs(64, 9, 8, 4), _obs(64, 9, 8, 4, fov=1.2, diameter=300.0), _obs(64, 7, 5, 2)]
    plans, Vs, Gs, As, rs = [], [], [], [], []
    for s, obs in enumerate(obs_list):
        A, vis = _random_problem(50 + s, obs)
        plans.append(idg_mod.Plan(obs, mac_unit=idg_mod.IDG_MAC_TENSOR))
        As.append(torch.as_tensor(A).cuda())
        Vs.append(torch.as_tensor(vis).cuda())
        Gs.append(torch.zeros((4, obs.grid_size, obs.grid_size), dtype=torch.complex128, device="cuda"))
    try:
        idg_mod.grid_many(plans, Vs, As, Gs)
        outs = [torch.zeros_like(v) for v in Vs]
        idg_mod.degrid_many(plans, Gs, As, outs)
        torch.cuda.synchronize()
        for p, V, A, G, o in zip(plans, Vs, As, Gs, outs):
            ref = torch.zeros_like(G)
            p.grid(V, A, ref)
            v = torch.zeros_like(V)
            p.degrid(G, A, v)
            p.synchronize()
            assert float(torch.linalg.vector_norm(G - ref) / torch.linalg.vector_norm(ref)) < 1e-12
            assert float((o - v).abs().max() / v.abs().max()) < 1e-6
    finally:
        for p in plans:
            p.close()
