"""The factored kernels hold values in pairs of halves with a power-of-two scale
each: correlations (and feeds) of very different strength keep their own
accuracy, and a value that is not finite stays in its correlation.

Tolerance 1e-5 of each plane's or correlation's own norm or maximum, as
elsewhere; the kernels' error is near 5e-7 whatever the strength."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_parity import DEGRID_TOL, GRID_TOL, Case, _degrid_err, _random_problem, _rel

pytestmark = pytest.mark.gpu

AMP = [(1.0, 1e-5, 1e-7, 1.0), (1e-8, 1.0, 1e4, 1e-3), (1e12, 1e-6, 1e-6, 1e-12)]


def _problem(L, amp, jones, seed=3):
    """Visibilities and model planes of the given strengths; diagonal A-terms, with the YY feed at 1e-4 of XX for
    "feeds", or full ones whose off-diagonal entries are so small that strength does not leak across correlations."""
    obs = synth.config(2, n_stations=8, n_timesteps=9, n_channels=7)
    A, vis = _random_problem(seed + L, obs, n_int=3)
    amp = np.array(amp)
    A[..., 1:3] = A[..., 1:3] * 1e-30 if jones == "full" else 0.0
    if jones == "feeds":
        A[..., 3] *= 1e-4
    rng = np.random.default_rng(seed)
    N = obs.grid_size
    G = (rng.standard_normal((4, N, N)) + 1j * rng.standard_normal((4, N, N))) * 1e-3 * amp[:, None, None]
    return obs, A.astype(np.complex64), (vis * amp).astype(np.complex64), G


@pytest.mark.parametrize("jones", ["diagonal", "feeds", "full"])
@pytest.mark.parametrize("amp", AMP)
@pytest.mark.parametrize("L", [32, 64, 96, 128])
def test_every_correlation_keeps_its_own_accuracy(idg_mod, oracle_mod, cuda_device, L, amp, jones):
    obs, A, vis, G = _problem(L, amp, jones)
    c = Case(idg_mod, oracle_mod, obs, A, vis, L=L, mac_unit=idg_mod.IDG_MAC_TENSOR)
    assert c.plan.kernels() == (idg_mod.IDG_KERNEL_FACTORED,) * 2
    got, ref = c.gpu_grid(), c.oracle_grid()
    for k in range(4):
        assert _rel(got[k], ref[k]) < GRID_TOL, k
    got, ref = c.gpu_degrid(G), c.oracle_degrid(G)
    for k in range(4):
        assert _degrid_err(got[..., k], ref[..., k]) < DEGRID_TOL, k


@pytest.mark.parametrize("L", [64, 96])
def test_mirrored_rows_keep_the_scale_of_their_correlation(idg_mod, cuda_device, L):
    """Rows of w < 0 are gridded as V^H, which swaps XY and YX: against the FP32 kernels, whose correlations are
    independent."""
    import torch
    from tests.test_gpu_many_kinds import _obs
    obs = _obs(L=L, heights=60.0, n_st=9)
    A, vis = _random_problem(L, obs)
    A[..., 1:3] = 0.0
    amp = np.array([1.0, 1e-7, 1e-3, 1.0])
    A, V = torch.as_tensor(A).cuda(), torch.as_tensor((vis * amp).astype(np.complex64)).cuda()
    res = []
    for mac in (idg_mod.IDG_MAC_TENSOR, idg_mod.IDG_MAC_FP32):
        plan = idg_mod.Plan(obs, flags=idg_mod.IDG_W_LAYERS, mac_unit=mac)
        try:
            assert plan.layers()[:, 1].any() and not plan.layers()[:, 1].all()
            G = torch.zeros(plan.grid_shape(), dtype=torch.complex128, device="cuda")
            plan.grid(V, A, G)
            out = torch.zeros_like(V)
            plan.degrid(res[0][0] if res else G, A, out)
            plan.synchronize()
            res.append((G, out, plan.kernels()))
        finally:
            plan.close()
    assert res[0][2] == (idg_mod.IDG_KERNEL_FACTORED,) * 2
    for k in range(4):
        a, b = res[0][0][:, k], res[1][0][:, k]
        assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) < GRID_TOL
        assert _degrid_err(res[0][1][..., k].cpu().numpy(), res[1][1][..., k].cpu().numpy()) < DEGRID_TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("k", [0, 1, 3])
def test_a_value_that_is_not_finite_stays_in_its_correlation(idg_mod, cuda_device, bad, k):
    """Diagonal A-terms keep correlations apart: those beside the bad one, of strengths a half cannot hold without a
    scale, come out as without it."""
    import torch
    obs, A, vis, G = _problem(64, (3e6, 1e-9, 1e9, 1e-6), "diagonal")
    plan = idg_mod.Plan(obs, subgrid_size=64, mac_unit=idg_mod.IDG_MAC_TENSOR)
    try:
        Ad = torch.as_tensor(A).cuda()
        V, M = torch.as_tensor(vis).cuda(), torch.as_tensor(G).cuda()
        V2, M2 = V.clone(), M.clone()
        V2[3, 2, 1, k] = bad
        N = obs.grid_size
        x0, y0 = plan.subgrids()[0][5:7]
        M2[k, int(y0) + 9, int(x0) + 14] = bad
        others = [q for q in range(4) if q != k]
        grids = []
        for v in (V, V2):
            out = torch.zeros((4, N, N), dtype=torch.complex128, device="cuda")
            plan.grid(v, Ad, out)
            grids.append(out)
        outs = []
        for m in (M, M2):
            out = torch.zeros_like(V)
            plan.degrid(m, Ad, out)
            outs.append(out)
        plan.synchronize()
        assert not torch.isfinite(torch.view_as_real(grids[1][k])).all()
        assert not torch.isfinite(torch.view_as_real(outs[1][..., k])).all()
        for q in others:
            assert float(torch.linalg.vector_norm(grids[1][q] - grids[0][q]) / torch.linalg.vector_norm(grids[0][q])) < 1e-12
            assert torch.equal(outs[1][..., q], outs[0][..., q])
    finally:
        plan.close()
