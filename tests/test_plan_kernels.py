"""The kernels a plan reports (host-only plans)."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth


def _plan(idg_mod, flags=0, taper_user=None, irregular=False, **kw):
    obs = synth.config(2, n_stations=8, n_timesteps=6, n_channels=6)
    if irregular:
        obs.freqs = obs.freqs + np.linspace(0.0, 1.0, obs.n_channels) ** 2 * 2e5
    return idg_mod.Plan(obs, flags=flags | idg_mod.IDG_HOST_ONLY, taper_user=taper_user, **kw)


def test_kernels_follow_unit_and_options(idg_mod):
    F, T, P = idg_mod.IDG_KERNEL_FACTORED, idg_mod.IDG_KERNEL_TENSOR, idg_mod.IDG_KERNEL_FP32
    # a taper that leaves the corners of the field at full weight: no w range of these subgrids is small enough
    for kw, want in [(dict(), (F, F)), (dict(irregular=True), (F, F)), (dict(flags=idg_mod.IDG_STOKES_I), (F, F)),
                     (dict(flags=idg_mod.IDG_NORMALIZE_ATERM), (P, F)), (dict(mac_unit=idg_mod.IDG_MAC_FP32), (P, P)),
                     (dict(mac_unit=idg_mod.IDG_MAC_TENSOR_DEGRID), (P, F)), (dict(degrid_channels=2), (P, P)),
                     (dict(taper_user=np.ones(96)), (T, T)),
                     (dict(taper_user=np.ones(96), irregular=True), (P, T)),
                     (dict(taper_user=np.ones(96), flags=idg_mod.IDG_STOKES_I), (P, P))]:
        p = _plan(idg_mod, **kw)
        assert p.kernels() == want, kw
        p.close()


def test_null_arguments_are_refused(idg_mod):
    assert idg_mod.load().idg_plan_kernels(None, None, None) == 1
