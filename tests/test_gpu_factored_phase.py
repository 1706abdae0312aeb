"""What the factored phasors neglect, pixel by pixel: one visibility against
one pixel of the field, so that neither the taper nor other sources hide an
error, with subgrids of a small and of a wide w range."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth

pytestmark = pytest.mark.gpu

C = 299792458.0
# Rounding of one phasor product: two __sincosf (2^-21.2 each), FP32 phases up to 4.7 (2.4e-7 each), split operands
# (2^-22 each), the first-order product in halves (1e-3 x 2^-10), the accumulation's correction (1.4e-7 a chunk and,
# in the degridder, L / 16 chunks: 1.1e-6).
ROUNDING = 4e-6
INNER, OUTER = 3e-7 + ROUNDING, 1e-6 + ROUNDING   # |l|, |m| <= FOV / 4 and <= FOV / 3


def _plan(idg_mod, L, fov, x, n_bl=12, wide=4, n_t=12, flags=0):
    """The grid is one subgrid; `wide` of the baselines sweep w over +-x wavelengths, the others over +-0.1."""
    rng = np.random.default_rng(L)
    freqs = np.array([150e6, 151e6])
    uvw = np.zeros((n_bl, n_t, 3))
    uvw[:, :, :2] = rng.uniform(0.05, 0.9, (n_bl, 1, 2)) / fov * (C / 151e6)  # within the grid's middle cell
    uvw[:, :, 2] = np.linspace(-1.0, 1.0, n_t) * np.where(np.arange(n_bl) < wide, x, 0.1)[:, None] * (C / 151e6)
    n_st = n_bl + 1
    bl = np.array([(0, k + 1) for k in range(n_bl)], np.int32)
    plan = idg_mod.Plan(grid_size=L, subgrid_size=L, kernel_padding=12 if L == 32 else 18, image_size=fov,
                        n_stations=n_st, baselines=bl, uvw=uvw, freqs=freqs, aterm_offsets=np.array([0, 5, n_t], np.int32),
                        flags=flags)
    assert plan.kernels() == (idg_mod.IDG_KERNEL_FACTORED,) * 2
    assert plan.stats().n_subgrids == n_bl  # parts are the kernels' business, not the partition's
    A = synth.aterms_identity(2, n_st)
    lmn = (np.arange(L) - L // 2) * fov / L
    l, m = np.meshgrid(lmn, lmn)  # [j, i]
    n1 = np.sqrt(1 - l * l - m * m) - 1
    w = uvw[..., None, :] * (freqs / C)[:, None]  # [bl, t, ch, 3]
    t = (2.0 * np.arange(L) - L) / L
    beta = 0.35 * np.pi * (12 if L == 32 else 18)
    taper = np.i0(beta * np.sqrt(1 - t * t)) / np.i0(beta)
    return plan, A, w, l, m, n1, np.outer(taper, taper)


VALUES = (1.0, 0.5j, -1.0, -1j)   # of the correlations
GEOMETRIES = [(32, 0.35, 5.0), (32, 0.35, 35.0), (64, 0.5, 1.5), (64, 0.5, 8.0), (96, 0.5, 3.9), (96, 0.5, 5.7),
              (96, 0.5, 11.0), (96, 0.35, 40.0), (128, 0.5, 4.5), (128, 0.5, 11.0),
              # small fields: long w ranges in wavelengths, tables far below the range of half precision
              (96, 0.2, 110.0), (64, 0.1, 700.0), (96, 0.05, 3000.0), (32, 0.02, 12000.0), (128, 0.005, 250000.0)]


@pytest.mark.parametrize("L,fov,x", GEOMETRIES)
def test_gridder_pixel_phases(idg_mod, cuda_device, L, fov, x):
    """One visibility at a time, at the ends and inside of the w range: its subgrid image over the taper is its phasor."""
    import torch
    plan, A, w, l, m, n1, taper = _plan(idg_mod, L, fov, x)
    try:
        Ad = torch.as_tensor(A).cuda()
        r = np.maximum(abs(l), abs(m)) / fov
        for b, t, c in [(0, 0, 1), (1, 11, 1), (2, 11, 0), (3, 5, 0), (3, 6, 1), (8, 0, 1)]:
            vis = torch.zeros((*w.shape[:3], 4), dtype=torch.complex64, device="cuda")
            vis[b, t, c] = torch.tensor(VALUES)
            X = plan.subgrid_images(vis, Ad, 0)[b].cpu().numpy().astype(np.complex128)
            plan.synchronize()
            ph = np.exp(2j * np.pi * (w[b, t, c, 0] * l + w[b, t, c, 1] * m + w[b, t, c, 2] * n1)) * taper
            for k, v in enumerate(VALUES):
                err = np.abs(X[k] / v - ph) / taper
                assert err[r <= 0.25].max() < INNER and err[r <= 1 / 3].max() < OUTER
    finally:
        plan.close()


@pytest.mark.parametrize("L,fov,x", GEOMETRIES)
def test_degridder_pixel_phases(idg_mod, cuda_device, L, fov, x):
    """One pixel at a time: the visibilities over the taper are the pixel's phasors."""
    import torch
    plan, A, w, l, m, n1, taper = _plan(idg_mod, L, fov, x)
    try:
        Ad = torch.as_tensor(A).cuda()
        k = np.arange(L) - L // 2
        a = L // 4
        for di, dj in [(0, 0), (a, a), (-a, a // 2), (3, -a)]:
            i, j = L // 2 + di, L // 2 + dj
            # the centred transform of a pixel of value 1 / L^2 (the subgrid's inverse transform is not normalised)
            plane = np.exp(-2j * np.pi * (np.outer(k * dj, np.ones(L)) + np.outer(np.ones(L), k * di)) / L) / L ** 2
            G = torch.as_tensor(plane[None] * np.array(VALUES)[:, None, None]).cuda()
            V = torch.zeros((*w.shape[:3], 4), dtype=torch.complex64, device="cuda")
            plan.degrid(G, Ad, V)
            plan.synchronize()
            ph = np.exp(-2j * np.pi * (w[..., 0] * l[j, i] + w[..., 1] * m[j, i] + w[..., 2] * n1[j, i]))
            for q, v in enumerate(VALUES):
                # other pixels hold the rounding of the FP32 subgrid transform (6e-8 of the plane's norm each, shrunk by
                # the taper): 1e-7 of the plane's value, which counts where the pixel's own taper is small
                noise = 1e-7 / taper[j, i] if max(abs(di), abs(dj)) > 0 else 0.0
                d = np.abs(V[..., q].cpu().numpy() / v / taper[j, i] - ph)
                assert d.max() < INNER + noise
    finally:
        plan.close()
