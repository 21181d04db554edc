"""The one-launch paths of small batches against the general ones at their borders: the same
configurations in a batch that just fits a path and in one that is a configuration too large for it.
Neighbour lists agree bit for bit and in order; energies and forces to the rounding of FP32 networks
summed in two orders (about 20 roundings of terms of the size of the result: 2e-6 of the largest
atomic energy, 1e-5 of RMS for forces, 1e-4 per layer for the gradient as everywhere)."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu


def clusters(n_cfg, per, n_species, seed=1):
    """n_cfg open or periodic clusters of `per` atoms (a function of the index), 1.1 A and more apart."""
    rng = np.random.default_rng(seed)
    pos, off = [], [0]
    for c in range(n_cfg):
        n = per(c)
        k = int(np.ceil(max(n, 1) ** (1 / 3)))
        site = rng.permutation(k ** 3)[:n]
        x = np.stack([site // (k * k), site // k % k, site % k], 1) * 2.0 + rng.uniform(-0.4, 0.4, (n, 3))
        pos.append(x + rng.uniform(-3, 3, 3))
        off.append(off[-1] + n)
    pbc = (np.arange(n_cfg)[:, None] % 3 > np.arange(3)[None]).astype(np.uint8)   # 0 to 2 periodic directions
    cell = np.tile((np.eye(3) * 17.0).ravel(), (n_cfg, 1))
    n = off[-1]
    return W.System(np.asarray(off, np.int64), np.concatenate(pos), rng.integers(0, n_species, n).astype(np.int32), cell,
                    pbc, n_species)


@pytest.mark.parametrize("n_cfg,per,n_species", [
    (1024, lambda c: c % 4, 3),          # configurations at the limit, some empty
    (3, lambda c: (2000, 2095, 1)[c], 8),   # 4,096 atoms, then one configuration more
    (5, lambda c: (0, 1021, 1, 1026, 3)[c] if c < 4 else 2, 1),   # network rows at 2,048 and 2,050
])
def test_small_paths_match_the_general_ones(n_cfg, per, n_species):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    big = clusters(n_cfg + 1, lambda c: per(c) if c < n_cfg else 7, n_species)
    if n_cfg == 5:
        big = clusters(n_cfg, per, n_species)
    small = big.subset(range(big.n_cfg - 1))
    n = small.n_atoms
    desc = W.descriptor_params(n_species, 3.1, 8, 4, 4, zeta=8.0)
    archs = [W._mlp(desc.D, (24, 10)) for _ in range(n_species)]
    rng = np.random.default_rng(0)
    theta = torch.as_tensor(W.init_weights(rng, desc, archs, 0.5, 0.3), dtype=torch.float32, device="cuda")
    f_ref = torch.as_tensor(rng.normal(size=(big.n_atoms, 3)), dtype=torch.float32, device="cuda")
    got = []
    for system in (small, big):
        pot, sysd = P.Potential(desc, archs), P.DeviceSystem(system)
        off, j, sh = pot.neighbors(sysd)
        E, Ea, F, V = pot.energy_forces(sysd, theta)
        # dF only on the atoms that both batches hold: the same parameter gradient
        u = f_ref[:system.n_atoms].clone()
        u[n:] = 0
        g = pot.param_vjp(sysd, theta, None, u)
        m = int(off[n])
        got.append([t.cpu().numpy() for t in (off[:n + 1], j[:m], sh[:m], Ea[:n], F[:n], g)])
    for a, b in zip(got[0][:3], got[1][:3]):
        np.testing.assert_array_equal(a, b)
    (ea, fa, ga), (eb, fb, gb) = got[0][3:], got[1][3:]
    rms = np.sqrt((fb.astype(np.float64) ** 2).mean())
    errs = (np.abs(ea - eb).max() / np.abs(eb).max(), np.abs(fa - fb).max() / rms,
            max(H.layer_errors(archs, ga.astype(np.float64), gb.astype(np.float64))))
    print("%d atoms: E %.3g, F %.3g, gradient %.3g" % (n, *errs))
    assert errs[0] <= 2e-6 and errs[1] <= 1e-5 and errs[2] <= H.TOL_DTHETA
