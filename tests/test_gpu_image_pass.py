"""The pass beside the master-grid transforms against the centred transforms written out in NumPy: grid sizes
that are and are not multiples of four (the pass takes mirrored pixels and the ones N/2 away together, with
classes of fewer pixels on the axes and in the middle), one plane and four, one w layer and several, and the
image in the grid's own buffer.

Tolerance.  Both sides are FP64: a transform of N^2 <= 17424 points is good to about eps log2(N^2) = 3e-15
relative, the phase 2 pi w0 n' (below 500 rad) to 500 eps = 1e-13, and the FP64 sums of the gridded plane differ
by their order, 1e-15: 1e-12, of the taper-weighted image (Parseval) where the taper is divided out."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _case(idg_mod, oracle_mod, N, w_layers, stokes_i):
    rng = np.random.default_rng(N)
    enu = synth.stations_uniform_disk(rng, 6, 60.0)
    enu[:, 2] = rng.normal(0.0, 300.0 if w_layers else 1.0, enu.shape[0])
    obs = synth.make_observation(enu, 4, 2.0, np.linspace(140e6, 160e6, 4), 4, N, 32, 12, 0.5, name="image pass")
    flags = (idg_mod.IDG_W_LAYERS if w_layers else 0) | (idg_mod.IDG_STOKES_I if stokes_i else 0)
    plan = idg_mod.Plan(obs, flags=flags)
    geom = oracle_mod.Geometry(obs.grid_size, obs.subgrid_size, obs.kernel_padding, obs.image_size,
                               aterm_nodes=obs.aterm_nodes)
    st = plan.stats()
    layers = int(st.n_w_layers) if w_layers else 1
    w0 = [(int(st.w_layer_min) + i + 0.5) * float(st.w_layer_step) if w_layers else 0.0 for i in range(layers)]
    assert (layers > 1) == w_layers
    l = (np.arange(N) - N // 2) * obs.image_size / N
    n1 = np.sqrt(1.0 - l[None, :] ** 2 - l[:, None] ** 2) - 1.0
    return rng, obs, plan, oracle_mod.image_taper(geom), [2.0 * np.pi * w * n1 for w in w0]


def _centred(x, transform):
    return np.fft.fftshift(transform(np.fft.ifftshift(x, axes=(-2, -1))), axes=(-2, -1))


@pytest.mark.parametrize("w_layers", [False, True])
@pytest.mark.parametrize("stokes_i", [False, True])
@pytest.mark.parametrize("N", [130, 132])
def test_transforms_match_numpy(idg_mod, oracle_mod, cuda_device, N, w_layers, stokes_i):
    import torch
    rng, obs, plan, taper, phase = _case(idg_mod, oracle_mod, N, w_layers, stokes_i)
    npol, L2 = (1 if stokes_i else 4), obs.subgrid_size ** 2
    A = torch.as_tensor(synth.aterms_random(rng, obs.n_intervals, obs.n_stations, obs.aterm_nodes)).cuda()
    vis = torch.as_tensor(synth.random_visibilities(rng, obs).astype(np.complex64)).cuda()
    img = rng.standard_normal((npol, N, N)) + 1j * rng.standard_normal((npol, N, N))
    # image -> grid
    img_d = torch.as_tensor(img).cuda()
    G = torch.empty(plan.grid_shape(), dtype=torch.complex128, device="cuda")
    plan.predict(img_d, A, G, torch.empty_like(vis))
    plan.synchronize()
    want = np.stack([_centred(img / (L2 * taper) * np.exp(-1j * p), np.fft.fft2) for p in phase])
    got = G.cpu().numpy().reshape(want.shape)
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < TOL
    assert np.array_equal(img_d.cpu().numpy(), img)
    if not w_layers:  # one layer: the image may lie in the grid's buffer
        G.reshape(npol, N, N).copy_(img_d)
        plan.predict(G, A, G, torch.empty_like(vis))
        plan.synchronize()
        assert np.array_equal(G.cpu().numpy().reshape(want.shape), got)
    # grid -> image
    G.zero_()
    plan.grid(vis, A, G)
    plan.synchronize()
    g = G.cpu().numpy().reshape(want.shape)
    out = torch.empty_like(img_d)
    plan.invert(vis, A, G, out)
    plan.synchronize()
    ref = sum(_centred(x, np.fft.ifft2) * N * N * np.exp(1j * p) for x, p in zip(g, phase)) / L2
    assert np.linalg.norm(out.cpu().numpy() * taper - ref) / np.linalg.norm(ref) < TOL
    if not w_layers:
        assert np.linalg.norm(G.cpu().numpy().reshape(want.shape) - g) / np.linalg.norm(g) < TOL
    plan.close()
