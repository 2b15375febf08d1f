"""Callers' arrays in device memory: used in place where kernels can use them,
through staging buffers where they cannot, with the same bits either way."""
import ctypes

import numpy as np
import pytest

from paper_1310_2041_gb300 import learned, workloads as W

pytestmark = pytest.mark.gpu

MESH = (9, 18, 7)  # x, y, z
GRID = MESH[::-1]
CUDA_ERROR = 2  # HPF_ERR_CUDA


def densities(seed, channels):
    return np.random.default_rng(seed).uniform(0.2, 0.8, (channels,) + GRID).astype(np.float32)


def at_byte(a, shift):
    """A device copy of a that starts `shift` bytes into an allocation: (the allocation, its address)."""
    import torch
    raw = torch.zeros(a.nbytes + 64, dtype=torch.uint8, device="cuda")
    raw[shift:shift + a.nbytes] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda()
    torch.cuda.synchronize()
    return raw, raw.data_ptr() + shift


def network(hpf):
    net = hpf.Propagator(MESH)
    net.set_weights(learned.init_params(3))
    net.scale = 4.0
    return net


@pytest.mark.parametrize("shift", [0, 4, 2, 1])
def test_training_reads_device_arrays_at_any_address(hpf_gpu, shift):
    x, nxt = densities(1, 4), densities(2, 2)
    with network(hpf_gpu) as net:
        loss, grads = net.backward(x, nxt)
        net.train_step(x, nxt, 1e-3)
        weights = net.get_weights()
    (kx, px), (kn, pn) = at_byte(x, shift), at_byte(nxt, shift)
    with network(hpf_gpu) as net:
        g, got = np.empty_like(grads), ctypes.c_double()
        assert net.lib.hpf_prop_backward(net.h, px, pn, g.ctypes.data, ctypes.byref(got)) == 0
        assert net.lib.hpf_prop_train_step(net.h, px, pn, 1e-3, None) == 0
        assert got.value == loss and np.array_equal(g, grads)
        assert np.array_equal(net.get_weights(), weights)
    del kx, kn


@pytest.mark.parametrize("shift_in,shift_out", [(0, 0), (4, 8), (2, 0), (0, 2), (1, 3)])
def test_predictions_at_any_address(hpf_gpu, shift_in, shift_out):
    import torch
    x = densities(1, 4)
    with network(hpf_gpu) as net:
        want = net.forward(x)
        (keep, px), (out, po) = at_byte(x, shift_in), at_byte(np.zeros_like(want), shift_out)
        assert net.lib.hpf_prop_forward(net.h, px, po) == 0
        torch.cuda.synchronize()
        got = out[shift_out:shift_out + want.nbytes].cpu().numpy().view(np.float32).reshape(want.shape)
        assert np.array_equal(got, want)
        del keep


SEGMENT = 12 << 20  # a tensor of this size has an allocation of its own


def address_near_an_end(nbytes):
    """(an allocation, the address `nbytes` before its end)."""
    import torch
    raw = torch.zeros(SEGMENT, dtype=torch.uint8, device="cuda")
    return raw, raw.data_ptr() + SEGMENT - nbytes


def test_device_arrays_that_are_too_short_are_refused(hpf_gpu):
    """A state, a prediction or a training input whose allocation ends inside it
    is an error (the staging copies refused it); nothing is launched on it."""
    import torch
    w = W.diblock(33, 4, 3, 4.4, 4, 1.0)
    d = W.generate(w)
    n = w.n_beads
    raw, short = address_near_an_end(12 * n - 4)
    whole = torch.zeros((n, 3), device="cuda")
    with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        assert s.lib.hpf_get_state(s.h, short, whole.data_ptr(), None) == CUDA_ERROR
        assert s.lib.hpf_get_state(s.h, whole.data_ptr(), short, None) == CUDA_ERROR
        assert np.array_equal(s.get_state()[0], d["pos"])
        assert s.lib.hpf_get_state(s.h, raw.data_ptr() + SEGMENT - 12 * n, None, None) == 0
    last = raw[SEGMENT - 12 * n:].cpu().numpy().view(np.float32).reshape(n, 3)
    assert np.array_equal(last, d["pos"])
    assert not raw[:SEGMENT - 12 * n].any()
    x, nxt = densities(1, 4), densities(2, 2)
    xd, nd = torch.from_numpy(x).cuda(), torch.from_numpy(nxt).cuda()
    with network(hpf_gpu) as net:
        before = net.get_weights()
        for px, pn in ((short, nd.data_ptr()), (xd.data_ptr(), short)):
            assert net.lib.hpf_prop_train_step(net.h, px, pn, 1e-3, None) == CUDA_ERROR
            assert net.lib.hpf_prop_forward(net.h, px, pn) == CUDA_ERROR
        assert np.array_equal(net.get_weights(), before)
        net.train_step(xd, nd, 1e-3)
        stepped = net.get_weights()
    with network(hpf_gpu) as net:  # the refused steps do not count in Adam's bias correction
        net.train_step(x, nxt, 1e-3)
        assert np.array_equal(net.get_weights(), stepped)


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 1003])
def test_states_are_read_back_to_any_memory(hpf_gpu, n):
    """Device outputs that kernels can write in place, alone and side by side in
    one allocation, and those that take the copies: beside a host output,
    overlapping, unaligned."""
    import torch
    w = W.Workload("free", [(n, [0])], 8.0, 8, 1, [[0.0]], 0.1, field_every=2, steps=2)
    d = W.generate(w)
    with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
        s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])
        s.step(3)
        pos, vel, _ = s.get_state()

        def read(p, v):
            assert s.lib.hpf_get_state(s.h, p, v, None) == 0

        def buffers(words):
            raw = torch.full((words,), -7.0, device="cuda")
            torch.cuda.synchronize()
            return raw, raw.data_ptr()

        def floats(raw, first, count=3 * n):
            return raw[first:first + count].cpu().numpy()

        p, v, _ = s.get_state(torch.empty((n, 3), device="cuda"), torch.empty((n, 3), device="cuda"))
        assert np.array_equal(p.cpu(), pos) and np.array_equal(v.cpu(), vel)
        for gap in (0, 1):  # side by side in one allocation, velocities first
            raw, a = buffers(6 * n + gap + 2)
            read(a + 4 * (1 + 3 * n + gap), a + 4)
            assert np.array_equal(floats(raw, 1), vel.reshape(-1))
            assert np.array_equal(floats(raw, 1 + 3 * n + gap), pos.reshape(-1))
            assert floats(raw, 0, 1) == -7 and floats(raw, 6 * n + gap + 1, 1) == -7
            assert gap == 0 or floats(raw, 3 * n + 1, 1) == -7
        raw, a = buffers(6 * n)  # one alone
        read(a, None)
        assert np.array_equal(floats(raw, 0), pos.reshape(-1)) and np.all(floats(raw, 3 * n) == -7)
        read(None, a + 12 * n)
        assert np.array_equal(floats(raw, 0), pos.reshape(-1))
        assert np.array_equal(floats(raw, 3 * n), vel.reshape(-1))
        host = np.zeros((n, 3), np.float32)  # one on the host
        raw, a = buffers(3 * n)
        read(a, host.ctypes.data)
        assert np.array_equal(floats(raw, 0), pos.reshape(-1)) and np.array_equal(host, vel)
        raw, a = buffers(3 * n + 1)  # overlapping: velocities are copied last
        read(a, a + 4)
        assert floats(raw, 0, 1) == pos[0, 0] and np.array_equal(floats(raw, 1), vel.reshape(-1))
        raw, a = at_byte(np.zeros((2, n, 3), np.float32), 2)  # unaligned
        read(a, a + 12 * n)
        got = raw[2:2 + 24 * n].cpu().numpy().view(np.float32).reshape(2, n, 3)
        assert np.array_equal(got[0], pos) and np.array_equal(got[1], vel)
