"""Descriptor rows into a buffer of the caller that starts at any float: the same values as in an aligned one."""
import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W
from tests import gpu_common as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zeta", [50.0, 4.0])
@pytest.mark.parametrize("copies", [1, 64])
def test_rows_at_any_offset(copies, zeta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    one = H.triclinic_system()
    off = np.arange(copies + 1, dtype=np.int64) * one.n_atoms
    system = W.System(off, np.tile(one.pos, (copies, 1)), np.tile(one.species, copies), np.tile(one.cell, (copies, 1)),
                      np.tile(one.pbc, (copies, 1)), one.n_species)
    desc = W.descriptor_params(2, 5.0, 6, 8, 8, zeta=zeta)   # even sizes: pairs of values are stored together
    pot, sysd = P.Potential(desc, [W._mlp(desc.D, (16,)) for _ in range(2)]), P.DeviceSystem(system)
    n = system.n_atoms * desc.D
    want = pot.descriptors(sysd).reshape(-1)
    static = torch.empty(n, device="cuda")
    P.panna_descriptors_static(desc, sysd, static)
    for shift in (1, 2, 3):
        buf = torch.full((n + 4,), -7.0, device="cuda")
        P.panna_descriptors(pot.ctx, sysd, buf[shift:])
        assert torch.equal(buf[shift:shift + n], want)
        assert (buf[:shift] == -7.0).all() and (buf[shift + n:] == -7.0).all()
        P.panna_descriptors_static(desc, sysd, buf[shift:shift + n])
        assert torch.equal(buf[shift:shift + n], static)
