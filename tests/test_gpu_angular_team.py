"""The matrix forms with several warps per atom (batches below 1,216 atoms, FP32 networks) against one
warp per atom: the same configurations alone, in every size of the warps' team, and in a batch above the
limit.  Both sum the same rounds of pairs; the teams add up to 64 parts of a species block in another
order (64 * 2^-24 = 3.8e-6 of the block's maximum; the entries' sums of a force likewise, of terms up to
five times its size: 2e-5 of RMS)."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu

# (system, species, cutoff, sectors, shells, zeta), configurations of the small batches
CASES = [("edges", 3, 5.5, 9, 8, 50.0), ("tiny_cell", 1, 6.5, 16, 8, 50.0), ("mixed_pbc", 2, 6.0, 8, 5, 20.0),
         ("triclinic", 2, 6.0, 16, 7, 4.0)]
MAKE = {"edges": H.ragged_with_edges, "tiny_cell": H.tiny_cell_system, "mixed_pbc": H.mixed_pbc_system,
        "triclinic": H.triclinic_system}


def repeat(system, k):
    off = np.concatenate([[0]] + [system.atom_off[1:] + c * system.n_atoms for c in range(k)])
    return W.System(off.astype(np.int64), np.tile(system.pos, (k, 1)), np.tile(system.species, k),
                    np.tile(system.cell, (k, 1)), np.tile(system.pbc, (k, 1)), system.n_species)


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
def test_teams_match_one_warp_per_atom(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    name, S, rc, n_theta, n_r, zeta = case
    one = MAKE[name]()
    n = one.n_atoms
    desc = W.descriptor_params(S, rc, 12, n_theta, n_r, zeta=zeta)
    archs = [W._mlp(desc.D, (32, 16)) for _ in range(S)]
    theta = torch.as_tensor(W.init_weights(np.random.default_rng(2), desc, archs, 0.3, 0.1), dtype=torch.float32,
                            device="cuda")

    def run(k):
        pot = P.Potential(desc, archs)
        P.panna_set_tuning(pot.ctx, "descriptor", 5)
        P.panna_set_tuning(pot.ctx, "adjoint", 6)
        sysd = P.DeviceSystem(repeat(one, k))
        G = pot.descriptors(sysd)
        assert torch.equal(G, pot.descriptors(sysd))
        _, _, F, V = pot.energy_forces(sysd, theta)
        return [x[:m].cpu().numpy().astype(np.float64) for x, m in ((G, n), (F, n), (V, one.n_cfg))]

    G0, F0, V0 = run(1216 // n + 1)
    for k in sorted({1} | {max(1, (16 * 152 // t) // n) for t in (64, 32, 16, 8, 4, 2)}):
        if k * n >= 1216:
            continue
        G, F, V = run(k)
        err, (ferr, rms) = H.descriptor_error(G, G0, desc), H.force_error(F, F0)
        verr = float(np.abs(V - V0).max() / (np.abs(V0).max() + 1e-30))
        print("%s x %d (%d atoms): G %.3g, F %.3g, virial %.3g" % (name, k, k * n, err, ferr, verr))
        assert err <= 3.8e-6
        if n == 1:   # no net force on a one-atom lattice: terms of the size of virial / cutoff cancel
            assert np.abs(F).max() <= 2e-5 * np.abs(V0).max() / rc
        else:
            assert ferr <= 2e-5 and rms > 1e-6
        assert verr <= 2e-4
