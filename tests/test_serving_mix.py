"""Serving requests of different channel layouts together, and the device
memory a request is admitted by."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import serve, synth
from tests.test_serving import _req


def _irregular(req):
    f = req.obs.freqs
    req.obs.freqs = f + np.linspace(0.0, 1.0, len(f)) ** 2 * 2e5
    return req


def _footprint_problems():
    """Segments of one visibility up to whole subgrids; short and long baselines; every subgrid size."""
    for L, n_ch, n_t, steps, n_st in [(32, 1, 40, 1, 24), (32, 16, 16, 4, 24), (64, 1, 60, 1, 16), (64, 30, 48, 8, 16),
                                      (96, 1, 24, 2, 16), (96, 48, 6, 1, 16), (96, 24, 56, 4, 16), (128, 3, 40, 5, 12)]:
        rng = np.random.default_rng(L + n_ch)
        enu = synth.stations_uniform_disk(rng, n_st, 1000.0 if L == 32 else 3000.0)
        yield synth.make_observation(enu, n_t, 2.0, np.linspace(140e6, 170e6, n_ch), steps, 512 if L == 32 else 4096, L,
                                     12 if L == 32 else 18, 0.35 if L == 32 else 0.5)


def test_footprint_covers_the_staged_records(idg_mod):
    """The factored gridder stages 768 bytes per started chunk of 16 visibilities of a segment, the others 128 bytes
    a visibility: what a request counts for them covers both, and stays within a few times the larger."""
    for obs in _footprint_problems():
        req = serve.Request(0, "grid", obs, 0.0, synth.aterms_identity(obs.n_intervals, obs.n_stations))
        p = idg_mod.Plan(obs, flags=idg_mod.IDG_HOST_ONLY)
        assert p.kernels()[0] == idg_mod.IDG_KERNEL_FACTORED
        sg, seg = p.subgrids(), p.segments()
        n = (seg[:, 3] - seg[:, 2]) * (sg[seg[:, 0], 4] - sg[seg[:, 0], 3])
        held = max(768 * int(np.sum(-(-n // 16))), 128 * obs.n_vis)
        assert held <= serve.record_bytes(obs) <= 4 * held
        others = obs.n_vis * 32 + obs.grid_size ** 2 * 64
        assert serve.footprint_bytes(req) >= others + serve.record_bytes(obs)
        p.close()


@pytest.mark.gpu
def test_footprint_covers_the_plan(idg_mod, cuda_device):
    for obs in _footprint_problems():
        req = serve.Request(0, "grid", obs, 0.0, synth.aterms_identity(obs.n_intervals, obs.n_stations))
        p = idg_mod.Plan(obs)
        held = p.stats().device_bytes + obs.n_vis * 32 + obs.grid_size ** 2 * 64 + req.aterms.nbytes
        assert held <= serve.footprint_bytes(req)
        p.close()


@pytest.mark.gpu
def test_uniform_and_irregular_requests_share_waves(idg_mod, cuda_device):
    """Uniform and irregular channels run the same kernels and report the same unit, so a wave holds both; each
    result is that of the request served alone."""
    reqs = [_req(i, kind="grid" if i % 4 < 2 else "degrid", n_st=8 + i) for i in range(8)]
    for r in reqs[::2]:
        _irregular(r)
    mixed = serve.Server(hbm_budget_bytes=48 << 30, max_slots=8, mode="batched").run(reqs)
    assert all(r.status == "ok" for r in mixed)
    for r, m in zip(reqs, mixed):
        alone = serve.Server(hbm_budget_bytes=48 << 30, mode="plain").run([r])[0]
        d = np.abs(alone.output - m.output).max() / np.abs(alone.output).max()
        assert d < 1e-6
