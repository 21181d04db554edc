"""The matrix forms of the angular kernels (descriptor variant 5, adjoint variant 6) at the edges of
their tiles: sector and shell counts around 8 and 16, exponents on both sides of every rule, atoms with
0, 1, 2 and many neighbours, one to three species.

Tolerances.  FP32 forms: descriptors as everywhere (TOL_G); the adjoint is linear in its per-term
relative errors (about 5e-7), and a force sums terms up to 30 times its size: 2e-5 of RMS between two
kernels.  Fast forms: zeta 2^-22 from the hardware log2 (1.2e-5 at zeta = 50), so 3e-5 of the block
maximum for descriptors and 30 times 1.2e-5 of RMS, 5e-4, for forces."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu

SYSTEMS = {
    "edges": (H.ragged_with_edges, 3, 5.5),
    "tiny_cell": (H.tiny_cell_system, 1, 4.5),
    "mixed_pbc": (H.mixed_pbc_system, 2, 6.0),
    "triclinic": (H.triclinic_system, 2, 5.0),
}
# (system, sectors, shells, zeta, radial shells, eps)
SHAPES = [("edges", 8, 8, 50.0, 32, 1e-6), ("edges", 5, 3, 4.0, 7, 1e-6), ("edges", 9, 8, 33.0, 33, 1e-6),
          ("edges", 16, 7, 32.0, 16, 1e-6), ("mixed_pbc", 7, 5, 1.0, 5, 1e-6), ("mixed_pbc", 8, 8, 1.5, 8, 1e-6),
          ("mixed_pbc", 17, 9, 20.0, 64, 1e-6), ("mixed_pbc", 12, 8, 16.0, 12, 1e-4),
          ("tiny_cell", 8, 8, 50.0, 16, 1e-6), ("tiny_cell", 1, 1, 15.5, 1, 1e-6), ("triclinic", 8, 4, 64.0, 20, 0.0),
          ("triclinic", 16, 8, 17.5, 24, 1e-6)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%s-%dx%d-z%g" % s[:4])
def test_matrix_forms_match(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    name, n_theta, n_r, zeta, n_rad, eps = shape
    make, S, rc = SYSTEMS[name]
    system = make()
    desc = W.descriptor_params(S, rc, n_rad, n_theta, n_r, zeta=zeta, eps_theta=eps)
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(S)]
    theta = W.init_weights(np.random.default_rng(2), desc, archs, 0.3, 0.1)
    Go = O.batch(system, desc, archs, theta, want_G=True)["G"]
    pot = P.Potential(desc, archs)
    sysd = P.DeviceSystem(system)
    th = torch.as_tensor(theta, dtype=torch.float32, device="cuda")

    def forces(adjoint, mode):
        P.panna_set_angular_precision(pot.ctx, mode)
        P.panna_set_tuning(pot.ctx, "descriptor", 0)
        P.panna_set_tuning(pot.ctx, "adjoint", adjoint)
        _, _, F, V = pot.energy_forces(sysd, th, P.PANNA_MLP_FP32)
        return F.cpu().numpy().astype(np.float64), V.cpu().numpy()

    P.panna_set_tuning(pot.ctx, "descriptor", 5)
    for mode, tol in ((0, H.TOL_G), (2, 3e-5)):
        P.panna_set_angular_precision(pot.ctx, mode)
        G = pot.descriptors(sysd)
        assert torch.equal(G, pot.descriptors(sysd))       # sums in a fixed order
        err = H.descriptor_error(G.cpu().numpy().astype(np.float64), Go, desc)
        print("%s mode %d: descriptors %.3g" % (name, mode, err))
        assert err <= tol
    for mode, tol in ((0, 2e-5), (2, 5e-4)):
        F0, V0 = forces(0, 0 if mode == 0 else 2)
        F6, V6 = forces(6, mode)
        err, rms = H.force_error(F6, F0)
        verr = float(np.abs(V6 - V0).max() / (np.abs(V0).max() + 1e-30))
        print("%s mode %d: forces %.3g (rms %.3g), virial %.3g" % (name, mode, err, rms, verr))
        assert (err if rms > 1e-6 else np.abs(F6).max()) <= (tol if rms > 1e-6 else 1e-5)
        assert verr <= 10 * tol
