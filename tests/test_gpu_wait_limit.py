"""Waits of the kernels with factored phasors that run out: the call ends by
itself, with the MMAs and copies it had started complete, reports
IDG_ERR_TIMEOUT, and leaves the context and the plan usable."""
import numpy as np
import pytest

from paper_2502_17789_gb300 import synth
from tests.test_gpu_parity import _random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n_ch,n_t", [(32, 3, 9), (64, 17, 12), (96, 24, 16), (128, 5, 8)])
def test_waits_that_run_out(idg_mod, cuda_device, L, n_ch, n_t):
    """With a limit of 0 the first wait that is not already over gives up, in the middle of the pipelines; several
    items per block, one plan and several in one launch."""
    import torch
    obs = synth.config(2, n_stations=20, n_timesteps=n_t, n_channels=n_ch)
    A, vis = _random_problem(L, obs)
    plan = idg_mod.Plan(obs, subgrid_size=L, mac_unit=idg_mod.IDG_MAC_TENSOR)
    other = idg_mod.Plan(obs, subgrid_size=L, mac_unit=idg_mod.IDG_MAC_TENSOR)
    try:
        V, Ad = torch.as_tensor(vis).cuda(), torch.as_tensor(A).cuda()
        shape = (4, obs.grid_size, obs.grid_size)

        def results():
            G = torch.zeros(shape, dtype=torch.complex128, device="cuda")
            out = torch.zeros_like(V)
            plan.grid(V, Ad, G)
            plan.degrid(G, Ad, out)
            plan.synchronize()
            return G, out

        G0, out0 = results()
        plan.set_wait_limit(0)
        other.set_wait_limit(0)
        for call in (lambda: plan.grid(V, Ad, torch.zeros_like(G0)),
                     lambda: plan.degrid(G0, Ad, torch.zeros_like(V)),
                     lambda: idg_mod.grid_many([plan, other], [V, V], [Ad, Ad],
                                               [torch.zeros_like(G0), torch.zeros_like(G0)]),
                     lambda: idg_mod.degrid_many([plan, other], [G0, G0], [Ad, Ad],
                                                 [torch.zeros_like(V), torch.zeros_like(V)])):
            call()
            with pytest.raises(idg_mod.IdgError) as e:
                plan.synchronize()
            assert e.value.status == 7
        plan.set_wait_limit(2_000_000_000)
        G1, out1 = results()
        assert float(torch.linalg.vector_norm(G1 - G0) / torch.linalg.vector_norm(G0)) < 1e-12
        assert float((out1 - out0).abs().max() / out0.abs().max()) < 1e-6
    finally:
        plan.close()
        other.close()


def test_limits_out_of_range_are_refused(idg_mod, cuda_device):
    plan = idg_mod.Plan(synth.config(1, n_stations=4))
    try:
        for bad in (-1, 2_000_000_001):
            with pytest.raises(idg_mod.IdgError) as e:
                plan.set_wait_limit(bad)
            assert e.value.status == 1
    finally:
        plan.close()
