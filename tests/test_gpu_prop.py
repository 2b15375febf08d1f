"""The learned density propagator on the GPU against its CPU oracle, through the C ABI.

Network kernels (BF16 operands, FP32 accumulation) against the FP64 oracle
of oracle/propagator.py, twice.

First against the oracle fed what the kernels consume (tests/prop_bf16.py:
the oracle's conv, SiLU and their derivatives with the GPU's BF16 roundings
applied in between -- input features formed in FP32, weights, hidden
activations, loss and back-propagated gradients).  What is left is the FP32
accumulation order (about 1e-6 of a 432-term sum) and the rare hidden value
whose FP32 pre-activation lies on the other side of a BF16 rounding boundary
than the FP64 one: it moves by one BF16 step (2^-8 relative), so no output
or gradient element can move by more than 2^-8 of the largest one through a
single such flip, and their few random flips keep the norm error near
sqrt(p) 2^-8 ~ 1e-4.  Held to 5e-4 of the norm per output and per layer's
weight and bias gradients, 2^-8 of the largest element element-wise, the
loss to 5e-5.  A wrong bias, a swapped channel or a SiLU rounded the wrong
way fails these.

Second against the unrounded FP64 oracle: every BF16 rounding carries a
relative error of at most 2^-9; through three layers of 27 x 16-term sums
with mixed signs that is about 1e-2 of an output's norm, so outputs and
gradients are held to 3e-2 of their norm (and a cosine above 0.999),
FP32-only quantities (Adam) to FP32 rounding.

The learned MD step is checked by its two exact limits: a network with
zero weights predicts no change, and the learned window must then equal
the plain schedule with field_every = K bit for bit; a tolerance of zero
rejects every prediction, and the run must equal field_every = 1 bit for bit.
"""
import numpy as np
import pytest

import prop_bf16 as E
from oracle import propagator as P
from paper_1310_2041_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# ragged tiles, a mesh smaller than a tile, a mesh wrapping the box several
# times, and meshes large enough for the one-period wrap of the box copies
MESHES = [(13, 10, 5), (8, 8, 2), (3, 2, 2), (24, 16, 9), (20, 18, 19), (26, 34, 18)]


def rand_params(seed):
    rng = np.random.default_rng(seed)
    params = P.init_params(seed)
    # a last layer of ordinary size and non-zero biases, so every term matters
    params = [(W * (10.0 if k == 2 else 1.0), rng.normal(scale=0.2, size=b.shape))
              for k, (W, b) in enumerate(params)]
    return params


def rand_phi(shape, seed, c=4):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.0, 1.2, size=(c,) + shape)


def grid(mesh):
    return (mesh[2], mesh[1], mesh[0])


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


# bars against the BF16-emulated oracle (module docstring)
EMU_NORM = 5e-4
EMU_ELEM = 2.0 ** -8
EMU_LOSS = 5e-5


def within_emulated(got, ref, what):
    got = np.asarray(got, np.float64)
    assert rel(got, ref) < EMU_NORM, f"{what}: norm error {rel(got, ref):.2e}"
    err = np.max(np.abs(got - ref))
    assert err <= EMU_ELEM * np.max(np.abs(ref)), f"{what}: element error {err:.2e}"


def cosine(a, b):
    a = np.asarray(a, np.float64).ravel()
    b = np.asarray(b, np.float64).ravel()
    return float(a @ b / (np.linalg.norm(a) * np.linalg.norm(b)))


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "x".join(map(str, m)))
def test_forward_matches_oracle(hpf_gpu, mesh):
    params = rand_params(1)
    x = rand_phi(grid(mesh), 2)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        y = net.forward(x.astype(np.float32))
    ye, _, _, _ = E.forward(params, x)
    within_emulated(y, ye, "output")
    yo, _ = P.forward(params, x)
    assert y.shape == yo.shape
    assert rel(y, yo) < 3e-2
    assert cosine(y, yo) > 0.999
    assert np.max(np.abs(y - yo)) < 0.1 * np.max(np.abs(yo))


@pytest.mark.parametrize("mesh,rep", [((33, 35, 31), 2), ((9, 18, 7), 4)],
                         ids=["66x70x62", "36x72x28"])
def test_gradients_of_a_repeated_input(hpf_gpu, mesh, rep):
    # a periodic input repeated along every axis has the gradients of one copy; on
    # the larger mesh a weight-gradient CTA takes up to three tiles, ragged ones
    # among them.  rep^3 is a power of two, so the loss gradient d / V rounds alike
    # and only the FP32 accumulation order differs: the same bars
    params = rand_params(3)
    x = rand_phi(grid(mesh), 4).astype(np.float32)
    nxt = (x[2:] + 0.1 * rand_phi(grid(mesh), 5, 2)).astype(np.float32)
    big = tuple(rep * m for m in mesh)
    with hpf_gpu.Propagator(big) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        tile = (1, rep, rep, rep)
        loss, g = net.backward(np.tile(x, tile), np.tile(nxt, tile))
    lo, go = E.backward(params, x, nxt)
    assert abs(loss - lo) < EMU_LOSS * lo
    for (W, b), (Wo, bo) in zip(hpf_gpu.unpack_params(g), go):
        within_emulated(W, Wo, "weights")
        within_emulated(b, bo, "biases")


@pytest.mark.parametrize("ctas", [1, 3, 7])
def test_forward_does_not_depend_on_the_cta_split(hpf_gpu, ctas):
    # few CTAs: long sweeps through many columns, the accumulator ring wrapping
    # many times, runs of planes starting and ending inside columns
    mesh = (26, 34, 18)
    params = rand_params(6)
    x = rand_phi(grid(mesh), 7).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        y0 = net.forward(x)
        net.set_ctas(ctas)
        y1 = net.forward(x)
        net.set_ctas(0)
        y2 = net.forward(x)
    assert np.array_equal(y0, y1)
    assert np.array_equal(y0, y2)
    ye, _, _, _ = E.forward(params, x)
    within_emulated(y1, ye, "output")


@pytest.mark.parametrize("mesh", [(70, 70, 2), (13, 10, 5), (3, 2, 2)],
                         ids=lambda m: "x".join(map(str, m)))
@pytest.mark.parametrize("ctas", [1, 2])
def test_forward_split_on_thin_and_tiny_meshes(hpf_gpu, mesh, ctas):
    # Mz = 2: every run of input planes wraps in z and ends with a padding
    # plane past the padded array; a mesh smaller than one box in x and y
    params = rand_params(8)
    x = rand_phi(grid(mesh), 9).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        y0 = net.forward(x)
        net.set_ctas(ctas)
        y1 = net.forward(x)
    assert np.array_equal(y0, y1)
    ye, _, _, _ = E.forward(params, x)
    within_emulated(y1, ye, "output")


def test_sweep_waits_give_up_and_the_handle_stays_usable(hpf_gpu):
    # the first layer with its finished planes never signalled: every CTA's
    # bounded waits must run out (no hang), the timeout be reported once, the
    # tensor memory be released, and the next forward be unaffected
    mesh = (26, 34, 18)
    params = rand_params(10)
    x = rand_phi(grid(mesh), 11).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        y0 = net.forward(x)
        st, secs = net.selftest_timeout()
        assert st == 6, st  # HPF_ERR_TIMEOUT
        assert secs < 5.0
        y1 = net.forward(x)
        net.set_ctas(3)  # long sweeps: the abort path with slots waiting for releases
        st, _ = net.selftest_timeout()
        assert st == 6, st
        net.set_ctas(0)
        y2 = net.forward(x)
    assert np.array_equal(y0, y1)
    assert np.array_equal(y0, y2)


def window(a, c, r=3):
    """The periodic (2r + 1)^3 window of a planar mesh a [C][Mz][My][Mx]
    centred on c = (z, y, x): the receptive field of the three layers there."""
    idx = [np.arange(ci - r, ci + r + 1) % a.shape[1 + k] for k, ci in enumerate(c)]
    return a[:, idx[0]][:, :, idx[1]][:, :, :, idx[2]]


def test_forward_full_mesh_sampled(hpf_gpu):
    # the 70^3 mesh of the 1M-bead melt, launched as every forward is (one CTA
    # per SM): outputs on the faces, at column and row boundaries of the
    # sweep (x = 13 / 14, y = 7 / 8) and at random voxels against the emulated
    # oracle evaluated on each voxel's 7^3 receptive field
    mesh = (70, 70, 70)
    params = rand_params(3)
    x = rand_phi(grid(mesh), 4).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        y = net.forward(x)
    rng = np.random.default_rng(5)
    special = [0, 1, 7, 8, 13, 14, 27, 28, 55, 56, 63, 64, 68, 69]
    pts = [tuple(rng.choice(special, 3)) for _ in range(120)]
    pts += [tuple(rng.integers(0, 70, 3)) for _ in range(80)]
    got = np.array([y[:, z, yy, xx] for z, yy, xx in pts])
    want = np.array([E.forward(params, window(x, p))[0][:, 3, 3, 3] for p in pts])
    within_emulated(got, want, "sampled output")


def test_zero_weights_predict_no_change(hpf_gpu):
    mesh = (13, 10, 5)
    with hpf_gpu.Propagator(mesh) as net:
        y = net.forward(rand_phi(grid(mesh), 3).astype(np.float32))
    assert np.all(y == 0.0)


def test_weights_round_trip(hpf_gpu):
    vec = hpf_gpu.pack_params(rand_params(4))
    with hpf_gpu.Propagator((8, 8, 4)) as net:
        assert net.n_params == vec.size == 9538
        net.set_weights(vec)
        assert np.array_equal(net.get_weights(), vec)


@pytest.mark.parametrize("mesh", [(13, 10, 5), (24, 16, 9), (20, 18, 19)],
                         ids=lambda m: "x".join(map(str, m)))
def test_backward_matches_oracle(hpf_gpu, mesh):
    params = rand_params(5)
    x = rand_phi(grid(mesh), 6)
    nxt = rand_phi(grid(mesh), 7, c=2)
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        loss, g = net.backward(x.astype(np.float32), nxt.astype(np.float32))
    target = nxt - x[2:]
    Le, ge = E.backward(params, x, nxt)
    assert loss == pytest.approx(Le, rel=EMU_LOSS)
    got = hpf_gpu.unpack_params(g)
    for k, ((gW, gb), (eW, eb)) in enumerate(zip(got, ge)):
        within_emulated(gW, eW, f"layer {k} weight gradient")
        within_emulated(gb, eb, f"layer {k} bias gradient")
    Lo, go = P.backward(params, x, target)
    assert loss == pytest.approx(Lo, rel=2e-2)
    for k, ((gW, gb), (oW, ob)) in enumerate(zip(got, go)):
        assert rel(gW, oW) < 3e-2, f"layer {k} weights"
        assert cosine(gW, oW) > 0.999, f"layer {k} weights"
        assert rel(gb, ob) < 3e-2, f"layer {k} biases"


def test_scaled_network_matches_oracle(hpf_gpu):
    """With a change scale s the change channels enter times s and the
    prediction leaves divided by s; the loss is s^2 times the squared error.
    Inputs with changes of the size one MD step makes (about 1e-2)."""
    mesh = (24, 16, 9)
    s = 25.0
    params = rand_params(21)
    rng = np.random.default_rng(22)
    x = rand_phi(grid(mesh), 23)
    x[:2] = x[2:] - rng.uniform(-0.04, 0.04, size=x[2:].shape)
    nxt = x[2:] + rng.uniform(-0.04, 0.04, size=x[2:].shape)
    with hpf_gpu.Propagator(mesh) as net:
        assert net.scale == 1.0
        net.scale = s
        assert net.scale == s
        net.set_weights(hpf_gpu.pack_params(params))
        assert net.scale == s  # loading weights keeps the scale
        y = net.forward(x.astype(np.float32))
        loss, g = net.backward(x.astype(np.float32), nxt.astype(np.float32))
        for bad in (0.0, -1.0, float("inf"), float("nan")):
            with pytest.raises(hpf_gpu.HPFError):
                net.scale = bad
        assert net.scale == s
    ye, _, _, _ = E.forward(params, x, s)
    within_emulated(y, ye, "scaled output")
    Le, ge = E.backward(params, x, nxt, s)
    assert loss == pytest.approx(Le, rel=EMU_LOSS)
    for k, ((gW, gb), (eW, eb)) in enumerate(zip(hpf_gpu.unpack_params(g), ge)):
        within_emulated(gW, eW, f"layer {k} weight gradient (scaled)")
        within_emulated(gb, eb, f"layer {k} bias gradient (scaled)")
    yo, _ = P.forward(params, x, s)
    assert rel(y, yo) < 3e-2 and cosine(y, yo) > 0.999
    Lo, go = P.backward(params, x, nxt - x[2:], s)
    assert loss == pytest.approx(Lo, rel=2e-2)
    for k, ((gW, gb), (oW, ob)) in enumerate(zip(hpf_gpu.unpack_params(g), go)):
        assert rel(gW, oW) < 3e-2 and cosine(gW, oW) > 0.999, f"layer {k} weights"
        assert rel(gb, ob) < 3e-2, f"layer {k} biases"


def test_adam_matches_oracle(hpf_gpu):
    params = rand_params(8)
    mesh = (8, 8, 4)
    x = rand_phi(grid(mesh), 9)
    t = rand_phi(grid(mesh), 10, c=2) - x[2:]
    state = P.adam_state(params)
    cur = params
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(params))
        for it in range(3):
            _, grads = P.backward(cur, x, t)  # oracle gradients, given to both sides
            gvec = hpf_gpu.pack_params(grads)
            net.adam_step(gvec, 1e-2)
            cur, state = P.adam_step(cur, [tuple(np.asarray(a, np.float64) for a in gr)
                                           for gr in hpf_gpu.unpack_params(gvec)],
                                     state, lr=1e-2)
        got = net.get_weights()
    want = hpf_gpu.pack_params(cur)
    assert np.max(np.abs(got - want)) < 2e-6


def test_train_step_is_backward_then_adam(hpf_gpu):
    params = hpf_gpu.pack_params(rand_params(11))
    mesh = (13, 10, 5)
    x = rand_phi(grid(mesh), 12).astype(np.float32)
    nxt = rand_phi(grid(mesh), 13, c=2).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as a, hpf_gpu.Propagator(mesh) as b:
        a.set_weights(params)
        b.set_weights(params)
        for _ in range(3):
            la = a.train_step(x, nxt, 1e-3, want_loss=True)
            lb, g = b.backward(x, nxt)
            b.adam_step(g, 1e-3)
            assert la == lb
        assert np.array_equal(a.get_weights(), b.get_weights())


def test_training_on_gpu_fits_a_teacher(hpf_gpu):
    """A student trained by the GPU kernels learns the map of an oracle teacher network."""
    mesh = (16, 16, 16)
    teacher = rand_params(14)
    xs = [rand_phi(grid(mesh), 20 + k) for k in range(4)]
    nexts = [x[2:] + P.forward(teacher, x)[0] for x in xs]
    with hpf_gpu.Propagator(mesh) as net:
        net.set_weights(hpf_gpu.pack_params(P.init_params(15)))
        x32 = [x.astype(np.float32) for x in xs]
        n32 = [n.astype(np.float32) for n in nexts]
        first = np.mean([net.backward(x, n)[0] for x, n in zip(x32, n32)])
        for it in range(400):
            net.train_step(x32[it % 4], n32[it % 4], 3e-3)
        last = np.mean([net.backward(x, n)[0] for x, n in zip(x32, n32)])
    assert last < 0.1 * first


# ---------------------------------------------------------------- learned MD step

def melt(hpf, n_chains=400, mesh=10, **over):
    n = n_chains * 10
    box = (n / 3.0) ** (1.0 / 3.0)
    w = W.diblock(n_chains, 5, 5, box, mesh, 1.0, name="learned_melt")
    pp = w.params()
    pp.update(over)
    data = W.generate(w)
    return w, pp, data


def system(hpf, pp, data, step=0):
    s = hpf.System(hpf.make_params(**pp))
    s.set_state(data["pos"], data["vel"], data["type"], data["bonds"], step)
    return s


def test_density_phi_is_the_scaled_mesh(hpf_gpu):
    w, pp, data = melt(hpf_gpu)
    s = system(hpf_gpu, pp, data)
    D = s.scatter_density()
    phi = s.density_phi()
    h = [np.float64(np.float32(pp["box"][a])) / pp["mesh"][a] for a in range(3)]
    phi_c = 2.0 ** -39 / (pp["rho0"] * (h[0] * h[1] * h[2]))
    assert np.array_equal(phi, (D.astype(np.float64) * phi_c).astype(np.float32))
    # mass conservation: every bead adds 1 / (rho0 h^3) in total
    vol = h[0] * h[1] * h[2]
    assert np.sum(phi, dtype=np.float64) * pp["rho0"] * vol == pytest.approx(w.n_beads, rel=1e-6)


def test_judge_matches_oracle_forces(hpf_gpu, orc):
    w, pp, data = melt(hpf_gpu)
    s = system(hpf_gpu, pp, data)
    phi = s.density_phi().astype(np.float64)
    rng = np.random.default_rng(3)
    cand = np.clip(phi + rng.normal(scale=0.1, size=phi.shape), 0.0, None).astype(np.float32)
    eps = s.judge_density(cand)
    assert s.judge_density(phi.astype(np.float32)) < 1e-5
    # the oracle: field forces of the candidate mesh and of the true mesh
    op = orc.make_params(**pp)
    h = [np.float64(np.float32(pp["box"][a])) / pp["mesh"][a] for a in range(3)]
    inv_phi_c = 1.0 / (2.0 ** -39 / (pp["rho0"] * (h[0] * h[1] * h[2])))
    Dc = np.maximum(np.rint(cand.astype(np.float64) * inv_phi_c), 0).astype(np.int64)
    Dt = orc.scatter(op, data["pos"], data["type"])
    Fc = orc.field_force(op, data["pos"], data["type"], orc.field(op, Dc)[1])
    Ft = orc.field_force(op, data["pos"], data["type"], orc.field(op, Dt)[1])
    eo = np.linalg.norm(Fc - Ft) / np.linalg.norm(Ft)
    assert eps == pytest.approx(eo, rel=1e-3)


def test_zero_network_equals_field_every_k(hpf_gpu):
    """Zero weights predict no change: after the first (plain) window every
    learned window runs the frozen field of its start, i.e. field_every = K."""
    K = 5
    w, pp, data = melt(hpf_gpu, field_every=1)
    a = system(hpf_gpu, pp, data)
    with hpf_gpu.Propagator((10, 10, 10)) as net:
        st = a.step_learned(net, 4, K=K, tol=1e9)
    assert st["windows"] == 4 and st["plain"] == 1 and st["learned"] == 3
    assert st["rejected"] == 0 and st["judged"] == 3
    # reference: K plain steps at field_every = 1, then field_every = K
    b = system(hpf_gpu, pp, data)
    b.step(K)
    pos, vel, step = b.get_state()
    ppk = dict(pp, field_every=K)
    c = system(hpf_gpu, ppk, {**data, "pos": pos, "vel": vel}, step)
    c.step(3 * K)
    pa, va, sa = a.get_state()
    pc, vc, sc = c.get_state()
    assert sa == sc == 4 * K
    assert np.array_equal(pa, pc) and np.array_equal(va, vc)


def test_zero_tolerance_equals_plain(hpf_gpu):
    """tol = 0 rejects every prediction: the run is field_every = 1 exactly."""
    K = 4
    w, pp, data = melt(hpf_gpu, field_every=1, sort_every=7)
    a = system(hpf_gpu, pp, data)
    with hpf_gpu.Propagator((10, 10, 10)) as net:
        net.set_weights(hpf_gpu.pack_params(P.init_params(2)))
        # window 1 builds history; window 2 is learned, rejected and re-run
        # plain; window 3 skips the judge (back-off 1), window 4 is judged aside
        # and fails (back-off 2), window 5 skips
        st = a.step_learned(net, 5, K=K, tol=0.0)
        assert (st["plain"], st["rejected"], st["learned"], st["judged"]) == (4, 1, 0, 2)
        # window 6 still skips; window 7's shadow judgement passes and switches
        # back to learned windows ...
        st = a.step_learned(net, 2, K=K, tol=1e9)
        assert (st["plain"], st["judged"], st["learned"]) == (2, 1, 0)
        # ... which a zero tolerance rejects again (window 8), window 9 skips
        st = a.step_learned(net, 2, K=K, tol=0.0)
        assert (st["rejected"], st["plain"], st["learned"], st["judged"]) == (1, 1, 0, 1)
    b = system(hpf_gpu, pp, data)
    b.step(9 * K)
    pa, va, sa = a.get_state()
    pb, vb, sb = b.get_state()
    assert sa == sb == 9 * K
    assert np.array_equal(pa, pb) and np.array_equal(va, vb)


def test_learned_window_judges_its_prediction(hpf_gpu):
    """The eps a learned window reports is the judge's error of D(t) + dphi
    against the true density at t + K (recomputed here through the ABI)."""
    K = 5
    w, pp, data = melt(hpf_gpu, field_every=1)
    a = system(hpf_gpu, pp, data)
    params = hpf_gpu.pack_params([(W * 0.3, b) for W, b in P.init_params(4)])
    with hpf_gpu.Propagator((10, 10, 10)) as net:
        net.set_weights(params)
        phi0 = a.density_phi()
        st = a.step_learned(net, 1, K=K, tol=1e9)       # plain window: history phi(0)
        assert st["plain"] == 1
        phiK = a.density_phi()
        dphi = net.forward(np.concatenate([phi0, phiK]))
        st = a.step_learned(net, 1, K=K, tol=1e9)       # learned window K .. 2K
        assert st["learned"] == 1
        eps = a.judge_density(phiK + dphi)
    # D(K) + dphi in the fixed point and phi(K) + dphi in FP32 differ by rounding only
    assert st["eps_last"] == pytest.approx(eps, rel=1e-3)
    assert 0.0 < eps < 10.0


def test_learned_window_in_one_launch_matches_per_step(hpf_gpu):
    """hpf_learned_mode: a learned window in one launch (the step kernel
    interpolating the fields of D(t) and D(t) + dphi) against one launch per
    step on the refreshed fixed-point meshes D(t) + (j/K) dphi.  The field is
    linear in the density, so the two differ by rounding only: the same
    windows accepted, the same judged eps to 1e-3, trajectories within the
    trajectory bar (1e-4)."""
    K = 6
    w, pp, data = melt(hpf_gpu, field_every=1)
    params = hpf_gpu.pack_params([(W * 0.3, b) for W, b in P.init_params(4)])
    out = []
    for in_launch in (True, False):
        a = system(hpf_gpu, pp, data)
        a.learned_mode(in_launch)
        with hpf_gpu.Propagator((10, 10, 10)) as net:
            net.set_weights(params)
            st = a.step_learned(net, 4, K=K, tol=1e9)
        out.append((st, a.get_state()))
        a.close()
    (s1, (p1, v1, t1)), (s2, (p2, v2, t2)) = out
    assert s1["learned"] == s2["learned"] == 3 and t1 == t2 == 4 * K
    assert np.max(np.abs(p1 - p2)) <= 1e-4 and np.max(np.abs(v1 - v2)) <= 1e-4
    assert s1["eps_last"] == pytest.approx(s2["eps_last"], rel=1e-3)


def test_trained_network_beats_holding_the_last_density(hpf_gpu):
    """What the network gains over the method without it (holding the density
    of the last true update, i.e. a frozen field between updates): trained on
    the GPU on snapshots of a plain run, it predicts held-out density changes
    with a smaller error than predicting no change, and its field-force error
    at t + K is below the frozen field's on a continuation of the run."""
    import torch
    from paper_1310_2041_gb300 import learned
    K = 20
    n_chains = 10000  # 200,000 beads at rho0 = 3
    box = (20.0 * n_chains / 3.0) ** (1.0 / 3.0)
    w = W.diblock(n_chains, 10, 10, box, 40, 0.5, name="a10b10_200k")
    pp = dict(w.params(), field_every=1, sort_every=1000)
    data = W.generate(w)
    s = hpf_gpu.System(hpf_gpu.make_params(**pp))
    s.set_state(data["pos"], data["vel"], data["type"], data["bonds"])
    s.step(1000)
    snaps = learned.collect_snapshots(s, 120, K)
    ex = learned.triples(120)
    with hpf_gpu.Propagator((40, 40, 40)) as net:
        net.set_weights(learned.init_params(0))
        net.scale = learned.change_scale(snaps, ex[:100])
        learned.train(net, snaps, 1500, lr=2e-3, lr_final=2e-4, examples=ex[:100])
        val_net, val_zero, val_lin = learned.validation_loss(net, snaps, ex[100:])
        res = learned.judge_candidates(s, net, 8, K, lags=(K,))
    # at this lag linear extrapolation overshoots and is worse than holding
    assert val_net < 0.9 * min(val_zero, val_lin)
    assert np.mean(res["net"]) < 0.95 * np.mean(res["hold_net"])
    assert np.mean(res["net"]) < 0.95 * np.mean(res[f"linear_{K}"])
    assert np.allclose(res["hold_net"], res[f"hold_{K}"][-len(res["hold_net"]):])
    del torch


def test_scaled_network_learns_short_lag_extrapolation(hpf_gpu):
    """At a lag of 2 steps the density change is nearly linear in time; with
    the change scale the trained network reaches the accuracy of linear
    extrapolation (and far beats holding the last density)."""
    from paper_1310_2041_gb300 import learned
    K = 2
    n_chains = 10000
    box = (20.0 * n_chains / 3.0) ** (1.0 / 3.0)
    w = W.diblock(n_chains, 10, 10, box, 40, 0.5, name="a10b10_200k")
    pp = dict(w.params(), field_every=1, sort_every=1000)
    data = W.generate(w)
    s = hpf_gpu.System(hpf_gpu.make_params(**pp))
    s.set_state(data["pos"], data["vel"], data["type"], data["bonds"])
    s.step(1000)
    snaps = learned.collect_snapshots(s, 120, K)
    ex = learned.triples(120)
    with hpf_gpu.Propagator((40, 40, 40)) as net:
        net.set_weights(learned.init_params(0))
        net.scale = learned.change_scale(snaps, ex[:100])
        assert 20.0 < net.scale < 500.0
        learned.train(net, snaps, 1500, lr=2e-3, lr_final=2e-4, examples=ex[:100])
        val_net, val_zero, val_lin = learned.validation_loss(net, snaps, ex[100:])
    assert val_net < 1.1 * val_lin
    assert val_net < 0.3 * val_zero


def test_learned_step_rejects_bad_arguments(hpf_gpu):
    w, pp, data = melt(hpf_gpu)
    a = system(hpf_gpu, pp, data)
    with hpf_gpu.Propagator((10, 10, 12)) as wrong, hpf_gpu.Propagator((10, 10, 10)) as net:
        calls = [lambda: a.step_learned(wrong, 1, K=4),          # another mesh
                 lambda: a.step_learned(net, 1, K=1),            # K below 2
                 lambda: a.step_learned(net, 1, K=65),           # K above 64
                 lambda: a.step_learned(net, -1, K=4),           # negative count
                 lambda: a.step_learned(net, 1, K=4, tol=-1.0),
                 lambda: a.step_learned(net, 1, K=4, tol=float("nan"))]
        for call in calls:
            with pytest.raises(hpf_gpu.HPFError) as e:
                call()
            assert e.value.status == 1
        # nothing moved
        assert a.get_state()[2] == 0
        st = a.step_learned(net, 0, K=4)
        assert st["windows"] == 0 and st["steps"] == 0


def test_judge_three_species_against_oracle(hpf_gpu, orc):
    """The judge works for any species count (the learned step needs two)."""
    w = W.Workload("ternary_small", [(40, [0, 1, 2, 1]), (90, [2])], 7.0, 8, 3,
                   [[0, 1.2, 0.3], [1.2, 0, 0.8], [0.3, 0.8, 0]], 0.05, 3, 10)
    pp = w.params()
    data = W.generate(w)
    s = system(hpf_gpu, pp, data)
    phi = s.density_phi().astype(np.float64)
    assert phi.shape == (3, 8, 8, 8)
    rng = np.random.default_rng(9)
    cand = np.clip(phi + rng.normal(scale=0.1, size=phi.shape), 0.0, None).astype(np.float32)
    eps = s.judge_density(cand)
    op = orc.make_params(**pp)
    h = [np.float64(np.float32(pp["box"][a])) / pp["mesh"][a] for a in range(3)]
    inv_phi_c = 1.0 / (2.0 ** -39 / (pp["rho0"] * (h[0] * h[1] * h[2])))
    Dc = np.maximum(np.rint(cand.astype(np.float64) * inv_phi_c), 0).astype(np.int64)
    Dt = orc.scatter(op, data["pos"], data["type"])
    Fc = orc.field_force(op, data["pos"], data["type"], orc.field(op, Dc)[1])
    Ft = orc.field_force(op, data["pos"], data["type"], orc.field(op, Dt)[1])
    assert eps == pytest.approx(np.linalg.norm(Fc - Ft) / np.linalg.norm(Ft), rel=1e-3)
    with hpf_gpu.Propagator((8, 8, 8)) as net:
        with pytest.raises(hpf_gpu.HPFError):
            s.step_learned(net, 1, K=4)


def test_autoregressive_rollout(hpf_gpu):
    """The K-step rollout feeds each prediction back: its first step is one
    forward pass, its second a forward pass on (phi(t), prediction); a network
    with zero weights holds phi(t), so its judged error is the error of the
    held density at t + K (recomputed on an identical trajectory)."""
    import torch
    from paper_1310_2041_gb300 import learned
    w, pp, data = melt(hpf_gpu, field_every=1)
    a = system(hpf_gpu, pp, data)
    prev = torch.from_numpy(a.density_phi()).cuda()
    a.step(1)
    cur = torch.from_numpy(a.density_phi()).cuda()
    with hpf_gpu.Propagator((10, 10, 10)) as net:
        net.set_weights(hpf_gpu.pack_params([(W * 0.3, b) for W, b in P.init_params(6)]))
        net.scale = 40.0
        d1 = net.forward(torch.cat([prev, cur]).contiguous(), out=torch.empty_like(cur))
        p1 = cur + d1
        d2 = net.forward(torch.cat([cur, p1]).contiguous(), out=torch.empty_like(cur))
        assert torch.equal(learned.rollout(net, prev, cur, 1), p1)
        assert torch.equal(learned.rollout(net, prev, cur, 2), p1 + d2)
    K, n = 3, 4
    b = system(hpf_gpu, pp, data)
    with hpf_gpu.Propagator((10, 10, 10)) as zero:
        assert torch.equal(learned.rollout(zero, prev, cur, K), cur)
        eps = learned.judge_rollout(b, zero, n, K)
    assert len(eps) == n and all(np.isfinite(eps))
    c = system(hpf_gpu, pp, data)
    c.step(1)
    want = []
    for _ in range(n):
        held = c.density_phi()
        c.step(K)
        want.append(c.judge_density(held))
    assert eps == pytest.approx(want, rel=1e-12)


def test_rollout_feeds_predictions_back(hpf_gpu):
    """hpf_prop_rollout: K autoregressive steps in the library give the same
    bits as K forward passes with the sum phi + dphi done in FP32 outside, and
    one step is the network's prediction phi(t) + dphi at the emulated bars."""
    mesh = (13, 10, 5)
    params = rand_params(31)
    rng = np.random.default_rng(32)
    cur = rand_phi(grid(mesh), 33, c=2)
    prev = cur + rng.uniform(-0.03, 0.03, size=cur.shape)
    x = np.concatenate([prev, cur]).astype(np.float32)
    with hpf_gpu.Propagator(mesh) as net:
        net.scale = 20.0
        net.set_weights(hpf_gpu.pack_params(params))
        got = net.rollout(x, 3)
        a, b = x[:2].copy(), x[2:].copy()
        for _ in range(3):
            d = net.forward(np.concatenate([a, b]))
            a, b = b, (b + d).astype(np.float32)
        one = net.rollout(x, 1)
        with pytest.raises(hpf_gpu.HPFError):
            net.rollout(x, 0)
    np.testing.assert_array_equal(got, b)
    ye, _, _, _ = E.forward(params, x.astype(np.float64), 20.0)
    within_emulated(one - x[2:], ye, "one rollout step")


def test_smooth_phi_matches_oracle(hpf_gpu):
    """hpf_smooth_phi (FP32) against the oracle's binomial filter (FP64) on a
    ragged mesh, in place and out of place."""
    w = W.diblock(300, 5, 5, 11.0, 11, 1.0)
    d = W.generate(w)
    pp = w.params()
    pp["mesh"] = (13, 10, 5)
    rng = np.random.default_rng(41)
    phi = rng.uniform(0.0, 1.2, size=(2, 5, 10, 13)).astype(np.float32)
    with hpf_gpu.System(hpf_gpu.make_params(**pp)) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        for passes in (0, 1, 4):
            got = s.smooth_phi(phi, passes)
            ref = P.smooth(phi.astype(np.float64), passes)
            assert np.max(np.abs(got - ref)) <= 1e-6 * np.max(np.abs(ref)), passes
        import torch
        t = torch.from_numpy(phi).cuda()
        s.smooth_phi(t, 3, out=t)
        np.testing.assert_allclose(t.cpu().numpy(), P.smooth(phi.astype(np.float64), 3),
                                   rtol=0, atol=1e-6)


def test_judge_density_pair(hpf_gpu):
    """eps of a density against itself is zero; against the true density it
    is hpf_judge_density's eps (the reference taken through FP32 phi)."""
    w = W.diblock(400, 5, 5, 10.0, 10, 1.0)
    d = W.generate(w)
    with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        true = s.density_phi()
        rng = np.random.default_rng(43)
        cand = (true + rng.normal(0.0, 0.02, true.shape)).astype(np.float32)
        assert s.judge_density_pair(cand, cand) == 0.0
        e_pair = s.judge_density_pair(cand, true)
        e_true = s.judge_density(cand)
        assert e_true > 1e-3
        assert abs(e_pair - e_true) <= 1e-5 * e_true + 1e-7


def test_judge_density_pair_waits_for_the_field_it_restores(hpf_gpu):
    """The call synchronises: nothing of it, the refresh that puts the true
    density's field back among it (50 us and more on this mesh), is left on the
    stream when it returns, and that refresh's field is the true one."""
    import torch
    w = W.diblock(50, 5, 5, 192.0, 192, 1.0)
    d = W.generate(w)
    with hpf_gpu.System(hpf_gpu.make_params(**w.params()), stream=torch.cuda.Stream()) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        true = torch.empty(s.mesh_shape, device="cuda")
        s.density_phi(true)
        cand = true + 0.5
        torch.cuda.synchronize()
        want = s.forces(hpf_gpu.FORCE_FIELD)
        stream = torch.cuda.ExternalStream(s.stream)
        left = []
        for _ in range(3):
            assert s.judge_density_pair(cand, cand) == 0.0
            left.append(not stream.query())
        assert not any(left)
        assert np.array_equal(s.forces(hpf_gpu.FORCE_FIELD), want)


def force_pair(hpf, s, pp, cand):
    """The FP32 field forces of a candidate density and of the true one, as FP64."""
    h = [np.float64(np.float32(pp["box"][a])) / pp["mesh"][a] for a in range(3)]
    inv_phi_c = 1.0 / (2.0 ** -39 / (pp["rho0"] * (h[0] * h[1] * h[2])))
    Dc = np.maximum(np.rint(cand.astype(np.float64) * inv_phi_c), 0).astype(np.int64)
    D = s.scatter_density()
    s.field(D_in=Dc)
    Fc = s.forces(hpf.FORCE_FIELD).astype(np.float64)
    s.field(D_in=D)
    return Fc, s.forces(hpf.FORCE_FIELD).astype(np.float64)


@pytest.mark.parametrize("n", [1, 2, 3])
def test_judge_sums_in_fp64(hpf_gpu, n):
    """eps of a few beads from their FP32 forces to FP64 rounding: a bead's three
    squares enter each sum by one rounding each (2^-53 of it at most), so the
    root of the quotient is off by at most (3 n + 3 n) / 2 + 1/2 + 1 of them."""
    w = W.Workload("few", [(n, [0])], 5.0, 5, 1, [[0.0]], 0.5, field_every=1, steps=1)
    pp = w.params()
    worst = 0.0
    for seed in range(40):
        rng = np.random.default_rng(seed)
        d = W.generate(w)
        pos = rng.uniform(0.0, 5.0, (n, 3)).astype(np.float32)
        with hpf_gpu.System(hpf_gpu.make_params(**pp)) as s:
            s.set_state(pos, d["vel"], d["type"], d["bonds"])
            cand = (s.density_phi() + rng.uniform(0.0, 0.3, s.mesh_shape)).astype(np.float32)
            eps = s.judge_density(cand)
            Fc, Ft = force_pair(hpf_gpu, s, pp, cand)
            diff = (Fc - Ft).astype(np.longdouble)
            want = np.sqrt((diff ** 2).sum() / (Ft.astype(np.longdouble) ** 2).sum())
            worst = max(worst, float(abs(eps - want) / want))
    assert worst <= (3 * n + 1.5) * 2.0 ** -53 * 1.001


@pytest.mark.parametrize("n", [456 * 256 - 1, 456 * 256 + 1, 2 * 456 * 256 + 77])
def test_judge_counts_every_bead_once(hpf_gpu, n):
    """Beads at both ends of the grid's rounds, each judged by a candidate that
    differs from the true density around that bead alone: left out or counted
    twice it changes eps by its share of the few beads there, the FP32 forces'
    summation by 1e-12 at most."""
    w = W.Workload("free", [(n, [0])], 40.0, 40, 1, [[0.0]], 0.5, field_every=1, steps=1)
    pp, d = w.params(), W.generate(w)
    with hpf_gpu.System(hpf_gpu.make_params(**pp)) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        true = s.density_phi()
        order = s.order()
        for slot in sorted({0, 456 * 256 - 1, 456 * 256, 2 * 456 * 256, n - 1}):
            if slot >= n:
                continue
            cand = true.copy()
            x, y, z = np.floor(d["pos"][order[slot]]).astype(int) % 40
            cand[0, z, y, x] += 0.5
            eps = s.judge_density(cand)
            Fc, Ft = force_pair(hpf_gpu, s, pp, cand)
            want = np.linalg.norm(Fc - Ft) / np.linalg.norm(Ft)
            assert eps == pytest.approx(want, rel=1e-12)
            assert np.any(Fc[order[slot]] != Ft[order[slot]])
