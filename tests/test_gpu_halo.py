"""The two block sizes of the halo kernel against each other, bit for bit.

Chains longer than 64 beads are advanced by windows with recomputed rims: 256
threads a window up to a rim of 16 beads, 512 beyond.  With the field frozen
over 16 steps, one launch of 16 steps and launches of 2, 5 and 6 (rims of 2 to
48 beads with angles and dihedrals) do the same operations per bead, so
positions and velocities agree exactly, in or beside a rim, at the ends of
chains and of the bead array.
"""
import numpy as np
import pytest

from paper_1310_2041_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BONDED = {
    "bonds": {},
    "angles": {"angle_k": 4.0, "angle_cos0": -0.5},
    "dihedrals": {"angle_k": 4.0, "angle_cos0": -0.5, "dihedral_k": 0.5, "dihedral_n": 3},
}


@pytest.mark.parametrize("bonded", list(BONDED))
@pytest.mark.parametrize("chains,length", [(3, 65), (5, 100), (11, 233)])
def test_launch_lengths_give_the_same_bits(hpf_gpu, chains, length, bonded):
    box = float((chains * length / 3.0) ** (1.0 / 3.0))
    w = W.diblock(chains, length // 2, length - length // 2, box, max(4, round(box)), 1.0,
                  field_every=16, dt=0.004)
    d = W.with_bond_angles(w, W.generate(w))
    out = []
    for calls in ((16, 16), (2, 5, 6, 3) * 2):
        with hpf_gpu.System(hpf_gpu.make_params(**{**w.params(), **BONDED[bonded]})) as s:
            s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("bonded", list(BONDED))
@pytest.mark.parametrize("force_mode", [0, 1, 2])
def test_launch_lengths_give_the_same_bits_with_rounding_friction(hpf_gpu, force_mode, bonded):
    """gamma m and dt / m whose products round, every field force."""
    chains, length = 11, 133
    box = float((chains * length / 3.0) ** (1.0 / 3.0))
    w = W.diblock(chains, length // 2, length - length // 2, box, round(box), 1.0, field_every=16,
                  dt=0.004, gamma=0.7, mass=1.3)
    d = W.with_bond_angles(w, W.generate(w))
    out = []
    for calls in ((16, 16), (2, 5, 6, 3) * 2, (1,) * 32):
        with hpf_gpu.System(hpf_gpu.make_params(**{**w.params(), **BONDED[bonded],
                                                   "force_mode": force_mode})) as s:
            s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b, c in zip(*out):
        assert np.array_equal(a, b) and np.array_equal(a, c)
