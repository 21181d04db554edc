"""The angular kernels at the ends of what the descriptor's parameters may be, through the default choice of
kernels and against the oracle: shells without width (eta = 0), large eps_theta, where y_m passes below 0 and
above 1 (below 0 for sectors outside [0, pi] only).  Bounds as everywhere; the fast forms (angular
precision 2) carry about zeta 2^-22 per term, 1.2e-5 at zeta = 50, and a force sums terms up to 30 times its
size: 5e-4 of RMS."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu


def repeat(system, k):
    off = np.concatenate([[0]] + [system.atom_off[1:] + c * system.n_atoms for c in range(k)])
    return W.System(off.astype(np.int64), np.tile(system.pos, (k, 1)), np.tile(system.species, k),
                    np.tile(system.cell, (k, 1)), np.tile(system.pbc, (k, 1)), system.n_species)


# (zeta, eta, eps, sectors, shells)
LIMITS = [(4.0, 0.0, 1e-6, 8, 8), (50.0, 0.0, 1e-6, 16, 5), (2.0, 12.0, 0.5, 8, 8), (2.0, 12.0, 0.5, 9, 8),
          (3.0, 12.0, 0.5, 8, 5)]


@pytest.mark.parametrize("copies", [1, 51])       # below and above the limit of the teams of warps
@pytest.mark.parametrize("limits", LIMITS, ids=lambda s: "z%g-eta%g-eps%g" % s[:3])
def test_parameter_limits(limits, copies):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zeta, eta, eps, n_theta, n_r = limits
    one = H.triclinic_system()
    n = one.n_atoms
    desc = W.descriptor_params(2, 5.0, 8, n_theta, n_r, zeta=zeta, eta_ang=eta, eps_theta=eps)
    if eps > 0.1 and (n_theta, n_r) != (8, 8):
        desc = dataclasses.replace(desc, theta_s=np.linspace(-1.0, np.pi + 1.0, n_theta))
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(2)]
    rng = np.random.default_rng(2)
    theta = W.init_weights(rng, desc, archs, 0.3, 0.1).astype(np.float32)
    f_ref = rng.normal(size=(n, 3)).astype(np.float32)
    ref = O.batch(one, desc, archs, theta.astype(np.float64), want_G=True, e_ref=np.zeros(1),
                  f_ref=f_ref.astype(np.float64), w_force=1.0, param_grad=True)
    pot, sysd = P.Potential(desc, archs), P.DeviceSystem(repeat(one, copies))
    th = torch.as_tensor(theta, device="cuda")
    E_ref = torch.zeros(copies, dtype=torch.float64, device="cuda")
    F_ref = torch.as_tensor(np.tile(f_ref, (copies, 1)), device="cuda")
    for mode, tol_f in ((0, H.TOL_F_FP32), (2, 5e-4)):
        P.panna_set_angular_precision(pot.ctx, mode)
        _, _, F, _ = pot.energy_forces(sysd, th)
        _, g, _, _ = pot.loss_grad(sysd, th, E_ref, F_ref, 1.0)
        ferr, rms = H.force_error(F[:n].cpu().numpy().astype(np.float64), ref["F"])
        gerr = max(H.layer_errors(archs, g.cpu().numpy().astype(np.float64), ref["dtheta"]))
        print("mode %d: F %.3g (rms %.3g), gradient %.3g" % (mode, ferr, rms, gerr))
        assert ferr <= tol_f
        assert gerr <= H.TOL_DTHETA


@pytest.mark.parametrize("zeta", [20.0, 50.0])
def test_rows_with_large_eps(zeta):
    """eps = 3: y_m from -1/2 to 3/2."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    system = H.triclinic_system()
    desc = W.descriptor_params(2, 5.0, 8, 8, 8, zeta=zeta, eps_theta=3.0)
    archs = [W._mlp(desc.D, (16,)) for _ in range(2)]
    G0 = O.batch(system, desc, archs, np.zeros(2 * archs[0].n_params), want_G=True)["G"]
    pot = P.Potential(desc, archs)
    err = H.descriptor_error(pot.descriptors(P.DeviceSystem(system)).cpu().numpy().astype(np.float64), G0, desc)
    assert err <= H.TOL_G
