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
    desc = W.descriptor_params(2, 7.0, 8, 8, 8, zeta=zeta)                 # 48 neighbours: the forms differ by 2.3
    torch, archs, theta, th, pot, sysd = setup(repeat(one, 171), desc)     # 4,104 atoms
    ref = O.batch(one, desc, archs, theta.astype(np.float64))
    F = pot.energy_forces(sysd, th, P.PANNA_MLP_BF16)[2]
    choice = P.panna_tuning_choice(pot.ctx, "descriptor")
    assert (choice == 5) == matrix, choice
    err, _ = H.force_error(F[:one.n_atoms].cpu().numpy().astype(np.float64), ref["F"])
    assert err <= H.TOL_F_BF16


def clusters_of(n_species, copies, seed=7):
    """Boxes of 216 atoms on a jittered grid, about 18 neighbours within 3.2 A: with eight species 36 species
    blocks of four or five pairs each."""
    rng = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.0
    pos = g + rng.uniform(-0.35, 0.35, g.shape)
    one = W.System(np.array([0, 216], np.int64), pos, rng.integers(0, n_species, 216).astype(np.int32),
                   (np.eye(3) * 12.0).reshape(1, 9), np.ones((1, 3), np.uint8), n_species)
    return one, repeat(one, copies)


@pytest.mark.parametrize("copies", [1, 19])        # 216 and 4,104 atoms
@pytest.mark.parametrize("autotune", [1, 0])
@pytest.mark.parametrize("n_species", [5, 8])
def test_adjoint_of_many_species(n_species, autotune, copies):
    one, system = clusters_of(n_species, copies)
    desc = W.descriptor_params(n_species, 3.2, 8, 8, 8)
    torch, archs, theta, th, pot, sysd = setup(system, desc)
    P.panna_set_tuning(pot.ctx, "autotune", autotune)
    ref = O.batch(one, desc, archs, theta.astype(np.float64))
    for prec, tol in ((P.PANNA_MLP_FP32, H.TOL_F_FP32), (P.PANNA_MLP_BF16, H.TOL_F_BF16)):
        F = pot.energy_forces(sysd, th, prec)[2]
        choice = P.panna_tuning_choice(pot.ctx, "adjoint")
        if n_species == 8 and copies == 19:
            assert choice == 5, (prec, choice)      # 72 us against 257
        err, _ = H.force_error(F[:216].cpu().numpy().astype(np.float64), ref["F"])
        print("%d species, %d atoms, precision %d: variant %d, %.3g" % (n_species, 216 * copies, prec, choice, err))
        assert err <= tol


@pytest.mark.parametrize("rc,copies,n_theta,variant", [(3.2, 1, 8, 5), (5.6, 1, 8, 2), (5.6, 1, 16, 5), (5.6, 3, 8, 5)])
def test_tangent_of_small_dense_batches(rc, copies, n_theta, variant):
    """216 atoms with 18 and 87 neighbours, one and two chunks of sectors, and 648 with 87."""
    one, system = clusters_of(2, copies)
    desc = W.descriptor_params(2, rc, 8, n_theta, 8)
    torch, archs, theta, th, pot, sysd = setup(system, desc)
    f_ref = np.random.default_rng(3).normal(size=(216, 3)).astype(np.float32)
    ref = O.batch(one, desc, archs, theta.astype(np.float64), e_ref=np.zeros(1), f_ref=f_ref.astype(np.float64),
                  w_force=1.0, param_grad=True)
    g = pot.loss_grad(sysd, th, torch.zeros(copies, dtype=torch.float64, device="cuda"),
                      torch.as_tensor(np.tile(f_ref, (copies, 1)), device="cuda"), 1.0)[1]
    assert P.panna_tuning_choice(pot.ctx, "jvp") == variant
    assert max(H.layer_errors(archs, g.cpu().numpy().astype(np.float64), ref["dtheta"])) <= H.TOL_DTHETA
