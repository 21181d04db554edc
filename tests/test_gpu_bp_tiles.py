"""The BP kernels' tile sizes and passes: sector and shell counts on both sides of every rule, whole and
fractional exponents, atoms with no, one and many neighbours.  A force sums terms up to 30 times its
size, each to about 1e-6 (ten FP32 operations): 3e-5 of RMS; descriptors as everywhere (TOL_G); the
parameter gradient as everywhere (TOL_DTHETA)."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta,n_r", [(1, 1), (4, 2), (3, 4), (5, 3), (8, 5), (9, 2), (2, 9)])
@pytest.mark.parametrize("system", ["edges", "mixed_pbc"])
def test_bp_tiles(system, n_theta, n_r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sysm, S = (H.ragged_with_edges(), 3) if system == "edges" else (H.mixed_pbc_system(), 2)
    lam = np.where(np.arange(n_theta) % 2, -1.0, 1.0) * np.linspace(0.6, 1.0, n_theta)
    zeta = np.array([1.0, 2.5, 4.0, 16.0, 3.0])[np.arange(n_theta) % 5]
    desc = dataclasses.replace(W.descriptor_params(S, 5.0, 6, 1, 1), angular="bp", bp_lambda=lam, bp_zeta=zeta,
                               bp_eta=np.linspace(0.002, 0.08, n_r))
    archs = [W._mlp(desc.D, (16,)) for _ in range(S)]
    rng = np.random.default_rng(4)
    theta = W.init_weights(rng, desc, archs, 0.5, 0.05).astype(np.float32)
    e_ref, f_ref = rng.normal(size=sysm.n_cfg), rng.normal(size=(sysm.n_atoms, 3)).astype(np.float32)
    ref = O.batch(sysm, desc, archs, theta.astype(np.float64), want_G=True, e_ref=e_ref,
                  f_ref=f_ref.astype(np.float64), w_force=0.5, param_grad=True)
    pot, sysd = P.Potential(desc, archs), P.DeviceSystem(sysm)
    G = pot.descriptors(sysd)
    assert torch.equal(G, pot.descriptors(sysd))
    err = H.descriptor_error(G.cpu().numpy().astype(np.float64), ref["G"], desc)
    th = torch.as_tensor(theta, device="cuda")
    _, _, F, V = pot.energy_forces(sysd, th)
    ferr, rms = H.force_error(F.cpu().numpy().astype(np.float64), ref["F"])
    verr = np.abs(V.cpu().numpy() - ref["virial"]).max() / np.abs(ref["virial"]).max()
    _, g, _, _ = pot.loss_grad(sysd, th, torch.as_tensor(e_ref, device="cuda"), torch.as_tensor(f_ref, device="cuda"), 0.5)
    gerr = max(H.layer_errors(archs, g.cpu().numpy().astype(np.float64), ref["dtheta"]))
    print("%s %dx%d: G %.3g, F %.3g (rms %.3g), virial %.3g, dtheta %.3g" % (system, n_theta, n_r, err, ferr, rms,
                                                                            verr, gerr))
    assert err <= H.TOL_G
    assert ferr <= 3e-5
    assert verr <= 1e-4
    assert gerr <= H.TOL_DTHETA
