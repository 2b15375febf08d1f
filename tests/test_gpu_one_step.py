"""The one-step kernel against the field-period kernels, bit for bit.

With the field frozen over a period of four steps, four calls of one step go
through the one-step kernel and one call of four steps through the warp kernel
(chains of at most 64 beads) or the halo kernel (longer chains).  All form
every bead's update with the same operations in the same order, so positions
and velocities agree exactly.  Bead counts lie on both sides of the 256-bead
chunks and of the resident grid; chain lengths give segments that start on odd
beads and lanes whose second bead is another chain's.
"""
import numpy as np
import pytest

from paper_1310_2041_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def solvent_blend(chains, length, free, box, mesh):
    return W.Workload("blend", [(chains, [0] * length), (free, [1])], box, mesh, 2,
                      [[0.0, 1.0], [1.0, 0.0]], 0.1, field_every=4, steps=4)


SYSTEMS = {
    "one_bead": (W.diblock(1, 1, 0, 4.0, 4, 1.0, field_every=4), {}),
    "255": (W.diblock(15, 9, 8, 4.4, 4, 1.0, field_every=4), {}),
    "256_solvent": (solvent_blend(16, 15, 16, 4.4, 5), {}),
    "odd_chains": (W.diblock(301, 4, 3, 8.9, 9, 1.0, field_every=4), {}),
    "nve": (W.diblock(301, 4, 3, 8.9, 9, 1.0, field_every=4, gamma=0.0), {}),
    "andersen": (W.diblock(100, 7, 6, 7.6, 8, 1.0, field_every=4),
                 {"thermostat": 2, "andersen_nu": 20.0}),
    "long": (W.diblock(9, 40, 45, 6.3, 6, 1.0, field_every=4), {}),
    "long_andersen": (W.diblock(9, 40, 45, 6.3, 6, 1.0, field_every=4),
                      {"thermostat": 2, "andersen_nu": 20.0}),
    "200k": (W.diblock(10007, 9, 11, 40.6, 41, 1.0, field_every=4), {}),
}


@pytest.mark.parametrize("name", list(SYSTEMS))
def test_single_steps_give_the_bits_of_a_period(hpf_gpu, name):
    w, extra = SYSTEMS[name]
    d = W.generate(w)
    pos = (d["pos"] + 0.05 * np.random.default_rng(1).normal(size=d["pos"].shape)).astype(np.float32)
    out = []
    for calls in ((4, 4), (1,) * 8):
        with hpf_gpu.System(hpf_gpu.make_params(**{**w.params(), **extra})) as s:
            s.set_state(pos, d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("free", [127, 128, 129, 77824, 77825, 116737])
def test_chunk_sizes_give_the_bits_of_a_period(hpf_gpu, free):
    """Both sides of the small chunks' edges, of the system size up to which
    they are used and of the size one chunk per resident CTA covers."""
    w = solvent_blend(1, 7, free - 7, max(4.0, (free / 3.0) ** (1.0 / 3.0)), 4 if free < 200 else 32)
    d = W.generate(w)
    out = []
    for calls in ((4, 4), (1,) * 8):
        with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
            s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("chains", [3 * 304 - 1, 3 * 2432, 3 * 2432 + 1, 3 * 2700, 3 * 3300])
def test_rounds_of_segments_give_the_bits_of_single_steps(hpf_gpu, chains):
    """Three chains of 20 fill a segment: counts of segments below, at and
    beyond one round of the warps, with short and long last rounds."""
    w = W.diblock(chains, 9, 11, (chains * 20 / 3.0) ** (1.0 / 3.0), 30, 1.0, field_every=4)
    d = W.generate(w)
    out = []
    for calls in ((4, 4), (1,) * 8):
        with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
            s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("name", ["256_solvent", "odd_chains", "andersen", "long", "long_andersen", "200k"])
def test_friction_that_rounds_gives_the_bits_of_a_period(hpf_gpu, name):
    """gamma m and dt / m whose products round (above all factors are 1): every
    kernel fuses the friction with the field, so the bits still agree."""
    w, extra = SYSTEMS[name]
    d = W.generate(w)
    pos = (d["pos"] + 0.05 * np.random.default_rng(1).normal(size=d["pos"].shape)).astype(np.float32)
    out = []
    for calls in ((4, 4), (1,) * 8):
        with hpf_gpu.System(hpf_gpu.make_params(**{**w.params(), **extra, "gamma": 0.7, "mass": 1.3})) as s:
            s.set_state(pos, d["vel"], d["type"], d["bonds"])
            for n in calls:
                s.step(n)
            out.append(s.get_state() + (s.scatter_density(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
