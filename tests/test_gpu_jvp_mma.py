"""The tangent's matrix form (jvp variant 5) at the edges of its tiles: sector and shell counts around 8 and
16, exponents from the smallest it takes, atoms with 0, 1, 2 and many neighbours, one to three species.  The
training gradient is compared with variant 0's: both evaluate the terms to about zeta 2^-22 (hardware
logarithms; 1.2e-5 at zeta = 50), and the gradient's bound is 1e-4 of each layer's largest entry."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H
from tests.test_gpu_angular_mma import SHAPES, SYSTEMS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[3] >= 2] + [("mixed_pbc", 8, 8, 2.0, 8, 1e-6)],
                         ids=lambda s: "%s-%dx%d-z%g" % s[:4])
def test_matrix_form_matches(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    name, n_theta, n_r, zeta, n_rad, eps = shape
    make, S, rc = SYSTEMS[name]
    system = make()
    desc = W.descriptor_params(S, rc, n_rad, n_theta, n_r, zeta=zeta, eps_theta=eps)
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(S)]
    rng = np.random.default_rng(2)
    theta = torch.as_tensor(W.init_weights(rng, desc, archs, 0.3, 0.1), dtype=torch.float32, device="cuda")
    pot = P.Potential(desc, archs)
    sysd = P.DeviceSystem(system)
    u = torch.as_tensor(rng.normal(size=(system.n_atoms, 3)), dtype=torch.float32, device="cuda")
    E = torch.zeros(system.n_cfg, dtype=torch.float64, device="cuda")
    got = []
    for variant in (0, 5):
        P.panna_set_tuning(pot.ctx, "jvp", variant)
        got.append(pot.loss_grad(sysd, theta, E, u, 1.0)[1].cpu().numpy().astype(np.float64))
    assert np.isfinite(got[1]).all()
    err = max(H.layer_errors(archs, got[1], got[0]))
    print("%s: gradient %.3g" % (name, err))
    assert err <= 1e-4
