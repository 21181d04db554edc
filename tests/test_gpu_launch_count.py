"""panna_last_launch_count counts kernels: on the tensor cores a pair of back-products is two, on the CUDA cores one."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests.test_gpu_small_batches import clusters

pytestmark = pytest.mark.gpu


def test_pairs_of_back_products():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    system = clusters(42, lambda c: 50, 1)          # 2,100 rows: past the single-launch path
    desc = W.descriptor_params(1, 3.6, 8, 4, 4, zeta=16.0)
    arch = W._mlp(desc.D, (128, 128))               # one pair with 128 summands: through the second layer
    theta = torch.as_tensor(W.init_weights(np.random.default_rng(0), desc, [arch], 0.5, 0.3), dtype=torch.float32,
                            device="cuda")
    pot, sysd = P.Potential(desc, [arch]), P.DeviceSystem(system)
    E = torch.zeros(42, dtype=torch.float64, device="cuda")
    F = torch.zeros((2100, 3), device="cuda")
    count = []
    for path in (8, 12):                            # 8: the weight gradient only
        P.panna_set_tuning(pot.ctx, "mlp_fp32", path)
        pot.loss_grad(sysd, theta, E, F, 1.0)
        count.append(P.panna_last_launch_count(pot.ctx))
    assert count[1] == count[0] + 1
