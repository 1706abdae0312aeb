"""Each traffic capture's command makes a plan that runs the kernel it names
(host-only plans of the profiled workload)."""
import numpy as np
import pytest

import bench


@pytest.mark.parametrize("kern,place,kernel", [("gridder", 0, "IDG_KERNEL_FP32"), ("gridder_tc", 0, "IDG_KERNEL_TENSOR"),
                                               ("gridder_sep", 0, "IDG_KERNEL_FACTORED"),
                                               ("degridder", 1, "IDG_KERNEL_FP32"),
                                               ("degridder_tc", 1, "IDG_KERNEL_TENSOR"),
                                               ("degridder_sep", 1, "IDG_KERNEL_FACTORED")])
def test_capture_commands_reach_their_kernels(idg_mod, kern, place, kernel):
    from paper_2502_17789_gb300 import synth
    cmd = bench.ncu_traffic_command(kern)
    stations = int(cmd.split("--stations ")[1].split()[0])
    mac = int(cmd.split("--mac-unit ")[1].split()[0]) if "--mac-unit" in cmd else 0
    obs = synth.config(2, seed=0, n_stations=stations)
    plan = idg_mod.Plan(obs, flags=idg_mod.IDG_HOST_ONLY, mac_unit=mac,
                        taper_user=np.ones(obs.subgrid_size) if "--flat-taper" in cmd else None)
    assert plan.kernels()[place] == getattr(idg_mod, kernel)
    plan.close()
