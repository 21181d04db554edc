"""Which kernels the library takes by itself where a form is slower than another, and that the choice leaves results
as accurate as everywhere (BF16 networks: 1e-2 of RMS)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H
from tests.test_gpu_angular_limits import repeat

pytestmark = pytest.mark.gpu


def setup(system, desc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(desc.n_species)]
    theta = W.init_weights(np.random.default_rng(2), desc, archs, 0.3, 0.1).astype(np.float32)
    return torch, archs, theta, torch.as_tensor(theta, device="cuda"), P.Potential(desc, archs), P.DeviceSystem(system)


@pytest.mark.parametrize("zeta,matrix", [(6.0, False), (15.5, False), (16.0, True)])
def test_bf16_networks_below_the_fast_powers(zeta, matrix):
    one = H.triclinic_system()
    desc = W.descriptor_params(2, 5.0, 8, 8, 8, zeta=zeta)
    torch, archs, theta, th, pot, sysd = setup(repeat(one, 171), desc)     # 4,104 atoms
    ref = O.batch(one, desc, archs, theta.astype(np.float64))
    F = pot.energy_forces(sysd, th, P.PANNA_MLP_BF16)[2]
    choice = P.panna_tuning_choice(pot.ctx, "descriptor")
    assert (choice == 5) == matrix, choice
    err, _ = H.force_error(F[:one.n_atoms].cpu().numpy().astype(np.float64), ref["F"])
    assert err <= H.TOL_F_BF16
