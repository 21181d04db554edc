"""The matrix form of the descriptor below zeta = 16 (whole and fractional exponents) against 64 bits, next to the
blocked kernel: FP32 rows are no further off.  Both round the same ten or so operations per term, so one
system's errors differ by chance (by up to 15 % in the RMS over its rows); the geometric mean over four systems,
in teams of warps and with one warp per atom, has to be within a tenth."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H
from tests.test_gpu_angular_limits import repeat

pytestmark = pytest.mark.gpu

SYSTEMS = [(H.ragged_with_edges, 3, 5.5), (H.mixed_pbc_system, 2, 6.0), (H.triclinic_system, 2, 5.0),
           (lambda: H.triclinic_system(seed=8, n=30), 2, 6.0)]


@pytest.mark.parametrize("zeta", [1.0, 2.5, 4.0, 6.0, 10.3, 15.0, 15.5])
def test_rows_are_no_further_off(zeta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ratios = []
    for make, S, rc in SYSTEMS:
        one = make()
        desc = W.descriptor_params(S, rc, 8, 8, 8, zeta=zeta)
        archs = [W._mlp(desc.D, (16,)) for _ in range(S)]
        G0 = O.batch(one, desc, archs, np.zeros(sum(a.n_params for a in archs)), want_G=True)["G"]
        ang = slice(desc.n_species * desc.n_rad, None)
        scale = np.maximum(H.block_scales(desc, G0), 1e-6 * np.abs(G0).max())[ang]
        pot = P.Potential(desc, archs)
        for copies in (1, 1216 // one.n_atoms + 1):
            sysd, err = P.DeviceSystem(repeat(one, copies)), []
            for variant in (0, 5):
                P.panna_set_tuning(pot.ctx, "descriptor", variant)
                G = pot.descriptors(sysd)[:one.n_atoms].cpu().numpy().astype(np.float64)
                err.append(np.sqrt((((G - G0)[:, ang] / scale) ** 2).mean()))
            ratios.append(err[1] / err[0])
            assert H.descriptor_error(G, G0, desc) <= H.TOL_G
    print("zeta %g: %s" % (zeta, " ".join("%.2f" % r for r in ratios)))
    assert np.exp(np.log(ratios).mean()) <= 1.1
