"""The kernels that the bench line claims for its aperture measures are those that the device ran."""
import os
import sys

import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,n_phi,n_ap", [(2, 9, 3), (10, 129, 24), (4, 300, 64)])
def test_launches_of_the_aperture_measures(torch_cuda, nb, n_phi, n_ap):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch = torch_cuda
    from torch.profiler import ProfilerActivity, profile
    est = ext4pcf.Estimator(0, "f16x3")
    ups = torch.ones(est.ups_shape(nb, 3)[1:], dtype=torch.float64, device="cuda:0")
    args = (ups, np.geomspace(1.0, 9.0, nb + 1), n_phi, np.geomspace(1.0, 5.0, n_ap))
    est.to_map4(*args)
    torch.cuda.synchronize()
    for _ in range(2):  # (a process' first profile may come up empty)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            est.to_map4(*args)
            torch.cuda.synchronize()
    names = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA and "ext4pcf" in e.name]
    est.close()
    assert len(names) == bench.map4_launches(nb, n_phi, n_ap), names
