"""Plans of two devices in one process (a plan belongs to the device that was
current when it was made): what a kernel needs set per device is set on both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_fp64_plans_on_two_devices():
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    if torch.cuda.device_count() < 2:
        pytest.skip("needs two devices")
    rng = np.random.default_rng(0)
    K, nG = 512, 130
    M = rng.standard_normal((K, nG)) + 1j * rng.standard_normal((K, nG))
    E = np.eye(nG) + 0.4 / np.sqrt(nG) * M[:nG]
    out = []
    for d in (0, 1):
        with torch.cuda.device(d):
            dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
            with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], [0.0], 1e-3, precision="fp64") as plan:
                chi = plan.accumulate(0, dev(M), 1, K, dev(np.zeros(1)), dev(np.ones(K)))
                inv = plan.epsilon_inverse(0, dev(E[None]))
                plan.sync_status()
            out.append((chi.cpu().numpy(), inv.cpu().numpy()))
    assert all(np.array_equal(a, b) for a, b in zip(*out))
