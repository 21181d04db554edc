"""Rebuilds of the neighbour list during a run of dynamics: candidates that outgrow their capacity are reported,
and past 4,096 atoms, where the search takes its general path, the kept list gives the trajectory of a search
every step (bounds as for the small batches)."""
import math

import numpy as np
import pytest

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _run(torch, pot, system, theta, v, dt, skin, steps, temperature=0.0, friction=0.0):
    sysd = P.DeviceSystem(system)
    vel = torch.as_tensor(v, dtype=torch.float64, device="cuda").contiguous()
    F = torch.zeros((system.n_atoms, 3), dtype=torch.float32, device="cuda")
    E = torch.zeros(system.n_cfg, dtype=torch.float64, device="cuda")
    builds = P.panna_md_run(pot.ctx, sysd, vel, theta, P.PANNA_MLP_FP32, dt, temperature, friction, skin, [12.011], 11, 0,
                            steps, F, False, E)
    torch.cuda.synchronize()
    return sysd.pos.cpu().numpy(), builds


@pytest.mark.parametrize("steps", [6, 8])      # the rebuild in the last step, and before it
def test_candidates_that_outgrow_the_list_are_reported(steps):
    torch = _torch()
    # 150 atoms on a sphere of 7.2 A about one atom, moving inwards by 0.26 A a step; nothing acts on them.
    # After 6 steps (1.56 A > skin / 2) the list is rebuilt at 5.64 A: the centre then has 150 candidates
    # within 6 A, more than cap_c = 8 * 16 + 8, and still no neighbour within 3 A; the others have about 11.
    k = np.arange(150) + 0.5
    z, phi = 1.0 - 2.0 * k / 150, k * math.pi * (3.0 - math.sqrt(5.0))
    u = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
    pos = np.concatenate([np.zeros((1, 3)), 7.2 * u])
    for r, cut in ((5.0, 3.0), (7.2, 6.0)):
        d = np.linalg.norm(u[:, None] - u[None], axis=-1) * r
        assert ((d < cut).sum(1) - 1).max() <= (16 if cut == 3.0 else 136)
    system = W.System(np.array([0, 151], np.int64), pos, np.zeros(151, np.int32), np.zeros((1, 9)),
                      np.zeros((1, 3), np.uint8), 1)
    desc = W.descriptor_params(1, 3.0, 4, 4, 4)
    archs = [W._mlp(desc.D, (8,))]
    pot = P.Potential(desc, archs, 16)
    theta = torch.zeros(pot.P, dtype=torch.float32, device="cuda")
    v = np.concatenate([np.zeros((1, 3)), -0.26 * u])
    moved, builds = _run(torch, pot, system, theta, v, 1.0, 3.0, 5)
    assert builds == 1 and abs(np.linalg.norm(moved[1:], axis=1) - 5.9).max() < 1e-9
    with pytest.raises(P.PannaError) as e:
        _run(torch, pot, system, theta, v, 1.0, 3.0, steps)
    assert e.value.status == P.PANNA_ERR_NEIGHBOR_OVERFLOW


def test_kept_list_past_the_small_batches():
    torch = _torch()
    wl = W.make("carbon16")
    one, k = wl.system, 260
    off = np.arange(k + 1, dtype=np.int64) * one.n_atoms
    system = W.System(off, np.tile(one.pos, (k, 1)), np.tile(one.species, k), np.tile(one.cell, (k, 1)),
                      np.tile(one.pbc, (k, 1)), one.n_species)
    assert system.n_atoms > 4096
    theta = torch.as_tensor(wl.theta.astype(np.float32), device="cuda")
    v = np.random.default_rng(5).normal(0.0, math.sqrt(8.617333262e-5 * 300.0 * 9.648533212e-3 / 12.011),
                                        (system.n_atoms, 3))
    pot = P.Potential(wl.desc, wl.archs)
    a, na = _run(torch, pot, system, theta, v, 0.5, 0.3, 40, 300.0, 0.02)
    b, nb = _run(torch, pot, system, theta, v, 0.5, 0.0, 40, 300.0, 0.02)
    assert nb == 41 and 2 <= na < 20
    assert np.abs(a - b).max() <= 1e-6
