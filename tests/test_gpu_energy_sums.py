"""Energies of large boxes through the layer products on the tensor cores: errors that are the same for all atoms add
up in the sum, those of FP32 sums mostly cancel.  Over 36 networks the sum of 4,096 atomic energies may be off by
at most twice as much as with the CUDA cores (RMS, relative to the sum of the energies' sizes), both against the
network in 64 bits on the same descriptors; a single atom's error is about half of theirs."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests.test_gpu_layer_products import energies_64

pytestmark = pytest.mark.gpu


def test_sums_of_atomic_energies():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(0)
    g = np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.0
    pos = g + rng.uniform(-0.35, 0.35, g.shape)
    off = {0: [], 12: []}
    for S, shape in ((1, (16, 8, 8)), (1, (64, 16, 8)), (2, (16, 8, 8))):
        system = W.System(np.array([0, 4096], np.int64), pos, rng.integers(0, S, 4096).astype(np.int32),
                          (np.eye(3) * 32.0).reshape(1, 9), np.ones((1, 3), np.uint8), S)
        sysd = P.DeviceSystem(system)
        for act, zeta in ((W.ACT_GAUSSIAN, 16.0), (W.ACT_TANH, 50.0)):
            desc = W.descriptor_params(S, 4.6, *shape, zeta=zeta)
            for hidden in ((128, 32), (256, 128), (512, 256)):
                archs = [W._mlp(desc.D, hidden, act) for _ in range(S)]
                for seed in (0, 1):
                    theta = torch.as_tensor(W.init_weights(np.random.default_rng(seed), desc, archs, 0.3, 0.1),
                                            dtype=torch.float32, device="cuda")
                    pot = P.Potential(desc, archs)
                    P.panna_set_tuning(pot.ctx, "descriptor", 5)
                    E64 = energies_64(desc, archs, theta, pot.descriptors(sysd), system.species)
                    for path in off:
                        P.panna_set_tuning(pot.ctx, "mlp_fp32", path)
                        E = pot.energy_forces(sysd, theta, virial=False)[1].cpu().numpy().astype(np.float64)
                        off[path].append((E - E64).sum() / np.abs(E64).sum())
    rms = {p: float(np.sqrt(np.mean(np.square(v)))) for p, v in off.items()}
    print("sums off by %.3g (CUDA cores), %.3g (tensor cores)" % (rms[0], rms[12]))
    assert rms[12] <= 2.0 * rms[0]
