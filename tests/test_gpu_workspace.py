"""Device memory of a handle's workspace: what a call reserves, and calls where memory is short.

Free memory is read from the device; "short" is made by holding most of it in a tensor.  Sizes are chosen
so that the routes differ by tens of megabytes (reservations) or gigabytes (short memory).
"""
import contextlib
import gc

import numpy as np
import pytest

from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


def probe_of(wl, **kw):
    from paper_1101_3615_gb300 import Probe
    return Probe(wl.m0, wl.h, wl.dt, wl.nt, wl.pad, wl.src, wl.rec, wl.wavelet, **kw)


def workload(shape, nt, ns, nb, pad=20):
    rng = np.random.default_rng(2)
    wl = mini_config(2, shape=shape, nt=nt, ns=1, pad=pad, p=1)
    wl.src = np.stack([np.full(ns, 2), rng.integers(0, shape[1], ns)], 1).astype(np.int32)
    wl.trials = (rng.standard_normal((nb,) + tuple(shape)) * 0.05 * wl.m0.mean()).astype(np.float32)
    return wl


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def only(leave):
    """Most of the device memory held, `leave` bytes of it free."""
    gc.collect()
    torch.cuda.empty_cache()
    held = torch.empty(free() - leave, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def reserved(wl, one_level, call):
    p = probe_of(wl)
    if one_level:
        p.set_option("pipeline", 2)
        p.set_option("tblock", 1)
    call(p)                               # kernels loaded, inputs staged
    p = probe_of(wl)
    if one_level:
        p.set_option("pipeline", 2)
        p.set_option("tblock", 1)
    before = free()
    call(p)
    return before - free(), p.stats()["pipeline_forward"]


def test_nonlinear_forward_reserves_no_second_derivative(cuda_device):
    wl = workload((100, 100), 400, 40, 1)
    m = torch.tensor(wl.m0, device=cuda_device)
    out = torch.empty((40, 400, wl.rec.shape[0]), device=cuda_device)
    resident, route = reserved(wl, False, lambda p: p.forward_nonlinear(m, out=out))
    assert route == 1
    assert resident <= reserved(wl, True, lambda p: p.forward_nonlinear(m, out=out))[0] + 16 * MB


def test_forward_on_the_one_level_kernels_reserves_no_segments(cuda_device):
    """A grid that a cluster holds, with so many fields that the one-level kernels are taken."""
    wl = workload((285, 405), 60, 64, 4)
    y = torch.tensor(wl.trials, device=cuda_device)
    out = torch.empty((4, 64, 60, wl.rec.shape[0]), device=cuda_device)
    got, route = reserved(wl, False, lambda p: p.apply_F(y, out=out))
    assert route != 1
    assert got <= reserved(wl, True, lambda p: p.apply_F(y, out=out))[0] + 16 * MB


def test_forward_and_migration_in_turn_keep_their_workspace(cuda_device):
    """A grid on which the Born fields fit a cluster and the adjoint fields do not."""
    wl = workload((300, 460), 50, 1, 1)
    p = probe_of(wl)
    y = torch.tensor(wl.trials, device=cuda_device)
    d = p.apply_F(y)
    assert p.stats()["pipeline_forward"] == 1
    img = p.apply_Fadj(d)
    assert p.stats()["pipeline_adjoint"] != 1
    out, im2 = torch.empty_like(d), torch.empty_like(img)
    left = free()
    for _ in range(2):
        p.apply_F(y, out=out)
        assert free() == left
        p.apply_Fadj(d, out=im2)
        assert free() == left
    assert torch.equal(out, d) and torch.equal(im2, img)


@pytest.mark.parametrize("K", [1, 5])
def test_resident_migration_after_a_one_level_one(cuda_device, K):
    """The one-level workspace has one segment of Dtt and of injection, the resident kernels take two."""
    wl = workload((40, 52), 20, 3, 1, pad=4)
    p = probe_of(wl, ckpt_stride=K)
    p.set_option("shot_group", 1)
    d = torch.randn((1, 3, 20, wl.rec.shape[0]), device=cuda_device, generator=torch.Generator(cuda_device).manual_seed(1))
    ref = p.apply_Fadj(d)
    assert p.stats()["pipeline_adjoint"] != 1
    p = probe_of(wl, ckpt_stride=K)
    p.set_option("autotune", 0)
    p.apply_Fadj(d)
    assert p.stats()["pipeline_adjoint"] != 1
    p.set_option("autotune", 1)
    assert torch.equal(p.apply_Fadj(d), ref)
    assert p.stats()["pipeline_adjoint"] == 1


def test_calls_that_fit_on_the_one_level_kernels_only(cuda_device):
    """Two Dtt segments of the resident kernels do not fit, one of the one-level kernels does."""
    from paper_1101_3615_gb300 import apply_H_group
    wl = workload((100, 100), 401, 64, 1)
    y = torch.tensor(wl.trials, device=cuda_device)

    def handles():
        out = [probe_of(wl, ckpt_stride=400) for _ in range(2)]
        for p in out:
            p.set_option("shot_wave", 64)     # the caller's wave, not the planner's
        return out

    probes = handles()
    ref = probes[0].apply_H(y)
    assert probes[0].stats()["pipeline_forward"] == 1
    for o in apply_H_group(probes, [y, y]):
        assert rel(o, ref) < 1e-6
    assert probes[0].stats()["pipeline_forward"] == 1
    probes = handles()
    with only(3600 * MB):                     # one-level 2.4 GB, resident 4.7 GB
        for _ in range(2):
            assert rel(probes[0].apply_H(y), ref) < 1e-6
        assert probes[0].stats()["pipeline_forward"] != 1
    with only(4600 * MB):                     # the second model's 2.4 GB fit beside the first's, 4.7 + 4.7 do not
        for _ in range(2):
            for o in apply_H_group(probes, [y, y]):
                assert rel(o, ref) < 1e-6
        assert probes[0].stats()["pipeline_forward"] != 1


@pytest.mark.parametrize("pipeline", [None, 2])
def test_planned_waves_fit_with_receivers_on_every_row(cuda_device, pipeline):
    """The receiver injection of a segment (200 bands) is most of the workspace."""
    wl = workload((200, 200), 201, 64, 4)
    wl.rec = np.stack([np.arange(200), np.full(200, 100)], 1).astype(np.int32)
    y = torch.tensor(wl.trials, device=cuda_device)

    def handle():
        p = probe_of(wl, ckpt_stride=100)
        if pipeline:
            p.set_option("pipeline", pipeline)
        return p

    p = handle()
    ref = p.apply_H(y)
    assert p.stats()["shot_wave"] == 64
    p = handle()
    with only(4096 * MB):
        assert rel(p.apply_H(y), ref) < 1e-6
        assert p.stats()["shot_wave"] < 64


def test_out_of_memory_is_reported_once(cuda_device):
    """The status of the call that ran out; what comes next finds no error of it."""
    from paper_1101_3615_gb300 import ProbeError
    wl = workload((200, 200), 201, 64, 4)
    y = torch.tensor(wl.trials, device=cuda_device)
    p = probe_of(wl, ckpt_stride=100)
    p.set_option("shot_wave", 64)
    with only(512 * MB):
        with pytest.raises(ProbeError) as ei:
            p.apply_H(y)
        assert ei.value.status == -3
        z = y + 1.0
    p.apply_H(y)
    assert float((z - y).mean()) == pytest.approx(1.0)


def test_gradient_in_planned_waves(cuda_device):
    """The model of a gradient is prepared in the workspace that its sweeps run in, whatever wave is planned."""
    wl = workload((100, 100), 401, 64, 1)
    m = torch.tensor(wl.m0, device=cuda_device) * 1.01
    p = probe_of(wl, ckpt_stride=400)
    d = p.forward_nonlinear(m)
    ref = p.gradient(m, d)
    p = probe_of(wl, ckpt_stride=400)
    with only(3072 * MB):
        for _ in range(2):
            assert rel(p.gradient(m, d), ref) < 1e-6
            assert p.stats()["shot_wave"] < 64
        assert rel(p.forward_nonlinear(m), d) < 1e-6
