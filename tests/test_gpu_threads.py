"""Host threads with contexts and streams of their own, whose batches ask the same kernels for different amounts
of shared memory: every call works, with the results of the calls made one after the other."""
import threading

import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests.test_gpu_small_batches import clusters

pytestmark = pytest.mark.gpu


def test_threads_with_batches_of_different_sizes():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # 3,800 atoms in 950 configurations need 90 KB of shared memory for their cells, 40 atoms 2 KB
    batches = [(clusters(950, lambda c: 4, 2), 120), (clusters(1, lambda c: 40, 2), 40)] * 2
    desc = W.descriptor_params(2, 5.0, 8, 8, 8)
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(2)]
    theta = torch.as_tensor(W.init_weights(np.random.default_rng(0), desc, archs, 0.3, 0.1), dtype=torch.float32,
                            device="cuda")
    jobs = [(P.Potential(desc, archs, cap), P.DeviceSystem(system)) for system, cap in batches]
    want = [pot.energy_forces(sysd, theta)[0].cpu().numpy() for pot, sysd in jobs]
    errors, start = [], threading.Barrier(len(jobs))

    def work(k):
        try:
            pot, sysd = jobs[k]
            E = torch.zeros(sysd.n_cfg, dtype=torch.float64, device="cuda")
            F = torch.zeros((sysd.n_atoms, 3), dtype=torch.float32, device="cuda")
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()   # E and F are cleared on another stream
            start.wait()
            for _ in range(500):
                P.panna_energy_forces(pot.ctx, sysd, theta, P.PANNA_MLP_FP32, E, None, F, None, stream)
            stream.synchronize()
            assert np.array_equal(E.cpu().numpy(), want[k])
        except Exception as e:   # noqa: BLE001 -- reported by the main thread
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
