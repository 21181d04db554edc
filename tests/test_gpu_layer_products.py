"""The FP32 networks' layer products on the tensor cores (mlp_fp32 = 12) against the CUDA cores' (0) past
the single-launch path: widths around 128 and 256, rows that are no multiple of a tile, species of a few
atoms and of none, descriptor widths that are no multiple of 4 (so no 16-byte loads).  The atomic energies
are compared with the network in 64 bits on the same descriptors: the tensor cores' error is not larger
than the CUDA cores' (their sums of 128 and more products carry 1.4 to 3 times the error).  Forces and
gradient are those of two FP32 networks summed in two orders: 1e-5 of RMS, 1e-4 per layer."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H
from tests.test_gpu_small_batches import clusters

pytestmark = pytest.mark.gpu

# (atoms, species in use, species, (n_rad, n_theta, n_r), hidden widths, activation)
CASES = [(2049, 1, 1, (64, 8, 8), (130, 129), W.ACT_GAUSSIAN), (2303, 2, 3, (7, 9, 5), (128, 257), W.ACT_TANH),
         (4100, 2, 2, (10, 6, 6), (256, 128, 16), W.ACT_GAUSSIAN), (2600, 3, 3, (32, 8, 8), (128, 32), W.ACT_GAUSSIAN)]


def energies_64(desc, archs, theta, G, species):
    """The networks in 64 bits on given descriptors."""
    import torch
    G, theta, E, at = G.double(), theta.double(), torch.zeros(len(species), dtype=torch.float64, device="cuda"), 0
    species = torch.as_tensor(species, device="cuda")
    for s, arch in enumerate(archs):
        h = G[species == s]
        for k, n, act in zip(arch.widths[:-1], arch.widths[1:], arch.acts):
            w, b = theta[at:at + n * k].view(n, k), theta[at + n * k:at + n * k + n]
            at += n * k + n
            h = h @ w.T + b
            h = {W.ACT_GAUSSIAN: lambda z: torch.exp(-z * z), W.ACT_TANH: torch.tanh, W.ACT_LINEAR: lambda z: z}[act](h)
        E[species == s] = h[:, 0]
    return E.cpu().numpy()


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%d-%d" % (c[0], c[2]))
def test_tensor_core_products_match_the_cuda_cores(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, used, S, shape, hidden, act = case
    system = clusters(n // 50 + 1, lambda c: 50 if c < n // 50 else n % 50, used)
    system.n_species = S
    if used == 3:
        system.species[3:] = np.where(system.species[3:] == 2, 0, system.species[3:])   # at most three atoms of it
    desc = W.descriptor_params(S, 3.6, *shape, zeta=16.0)
    archs = [W._mlp(desc.D, hidden, act) for _ in range(S)]
    rng = np.random.default_rng(0)
    theta = torch.as_tensor(W.init_weights(rng, desc, archs, 0.5, 0.3), dtype=torch.float32, device="cuda")
    E_ref = torch.as_tensor(rng.normal(size=system.n_cfg) * 10, dtype=torch.float64, device="cuda")
    F_ref = torch.as_tensor(rng.normal(size=(n, 3)), dtype=torch.float32, device="cuda")
    got = []
    for path in (0, 12):
        pot, sysd = P.Potential(desc, archs), P.DeviceSystem(system)
        P.panna_set_tuning(pot.ctx, "mlp_fp32", path)
        _, Ea, F, _ = pot.energy_forces(sysd, theta)
        _, g, _, _ = pot.loss_grad(sysd, theta, E_ref, F_ref, 1.0)
        again = pot.loss_grad(sysd, theta, E_ref, F_ref, 1.0)[1]
        got.append([x.cpu().numpy().astype(np.float64) for x in (Ea, F, g)])
        if path:   # sums in a fixed order; the forces' atomics move the gradient by their rounding
            errs = H.layer_errors(archs, again.cpu().numpy().astype(np.float64), got[-1][2])
            assert max(errs) <= 1e-5
    (E0, F0, g0), (E1, F1, g1) = got
    P.panna_set_tuning(pot.ctx, "descriptor", 5)
    E = energies_64(desc, archs, theta, pot.descriptors(sysd), system.species)
    err0, err1 = [float(np.sqrt(((x - E) ** 2).mean() / (E ** 2).mean())) for x in (E0, E1)]
    ferr, rms = H.force_error(F1, F0)
    gerr = max(H.layer_errors(archs, g1, g0))
    print("%d atoms: E %.3g and %.3g, F %.3g, gradient %.3g" % (n, err0, err1, ferr, gerr))
    assert err1 <= 1.1 * err0
    assert rms > 1e-6 and ferr <= 1e-5
    assert gerr <= 1e-4
