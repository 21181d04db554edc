"""Infinite activations through the layer products on the tensor cores: the result of the CUDA cores, not NaN.  One
hidden unit's bias is infinite; its weights in the next layer are all negative (ReLU then gives 0 and the
energies are finite) or all positive (the energies are infinite)."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests.test_gpu_small_batches import clusters

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bias", [np.inf, np.nan])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
@pytest.mark.parametrize("width", [128, 131])      # 16-byte loads, and rows that are no multiple of four
def test_infinite_activations(width, sign, bias):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    system = clusters(42, lambda c: 50, 1)          # 2,100 rows: past the single-launch path
    desc = W.descriptor_params(1, 3.6, 8, 4, 4, zeta=16.0)
    arch = W.MLPArch((desc.D, width, 32, 1), (W.ACT_LINEAR, W.ACT_RELU, W.ACT_LINEAR))
    theta = W.init_weights(np.random.default_rng(0), desc, [arch], 0.5, 0.3)
    first = width * desc.D
    theta[first + 5] = bias
    at = first + width
    w2 = theta[at:at + 32 * width].reshape(32, width)
    w2[:, 5] = sign * (0.1 + np.abs(w2[:, 5]))
    at += 32 * width + 32
    theta[at:at + 32] = 0.1 + np.abs(theta[at:at + 32])
    th = torch.as_tensor(theta, dtype=torch.float32, device="cuda")
    got = []
    for path in (0, 4):
        pot, sysd = P.Potential(desc, [arch]), P.DeviceSystem(system)
        P.panna_set_tuning(pot.ctx, "mlp_fp32", path)
        E, Ea, _, _ = pot.energy_forces(sysd, th)
        got.append([x.cpu().numpy() for x in (E, Ea)])
    (E0, Ea0), (E1, Ea1) = got
    if bias == np.inf:
        assert np.isfinite(Ea0).all() if sign < 0 else (Ea0 == np.inf).all()
    assert np.allclose(Ea0, Ea1, rtol=1e-5, atol=1e-6, equal_nan=True)
    assert np.allclose(E0, E1, rtol=1e-5, atol=1e-5, equal_nan=True)
