"""The register-queue 3D kernels (the default) against the one-barrier-per-plane kernels, bit for bit.

Both evaluate every cell update in the same order, and the adjoint's imaging terms, added three steps
at a time, in the order of the single steps.  Chunks that end one plane into a 32-plane piece, tiles cut
by the grid in x and y, no sponge and a wide one, segments of 1 to 5 steps, plain and compensated images.
"""
import numpy as np
import pytest

from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,pad,nt,K,ns,nb,kahan,planes", [
    ((24, 20, 50), 5, 23, 0, 2, 2, True, 0),
    ((33, 17, 64), 0, 18, 4, 1, 1, True, 32),       # one plane in the last chunk, no sponge
    ((9, 31, 66), 12, 17, 5, 3, 3, False, 64),
    ((129, 8, 12), 1, 15, 1, 1, 1, True, 128),      # segments of one step
    ((40, 33, 70), 3, 21, 2, 2, 1, False, 32),
    ((70, 16, 60), 2, 16, 3, 1, 5, True, 0),
])
def test_queue_kernels_give_identical_bits(cuda_device, shape, pad, nt, K, ns, nb, kahan, planes):
    from paper_1101_3615_gb300 import Probe
    rng = np.random.default_rng(5)
    wl = mini_config(5, shape=shape, nt=nt, ns=1, pad=pad, p=1)
    n = np.array(shape)
    rec = np.unique(np.stack([rng.integers(0, v, 60) for v in shape], 1), axis=0)   # distinct cells
    wl.rec = np.concatenate([rec, [[0, 0, 0]], [n - 1]]).astype(np.int32)
    wl.rec = np.unique(wl.rec, axis=0)
    wl.src = np.stack([rng.integers(0, v, ns) for v in shape], 1).astype(np.int32)
    w = (rng.standard_normal(nt) + 1.0).astype(np.float32)
    y = torch.tensor((rng.standard_normal((nb,) + shape) * 0.05 * wl.m0.mean()).astype(np.float32), device=cuda_device)
    probes = []
    for old in (False, True):
        p = Probe(wl.m0, wl.h, wl.dt, nt, pad, wl.src, wl.rec, w, kahan=kahan, ckpt_stride=K)
        if planes:
            p.set_option("planes3d", planes)
        if old:
            p.set_option("pipeline", 0)
        probes.append(p)
    q, o = probes
    d = o.apply_F(y)
    assert torch.equal(q.apply_F(y), d)
    assert q.stats()["pipeline_forward"] == 4
    r = torch.tensor(rng.standard_normal(tuple(d.shape)).astype(np.float32), device=cuda_device) * d.abs().max()
    assert torch.equal(q.apply_Fadj(r), o.apply_Fadj(r))
    assert torch.equal(q.apply_H(y), o.apply_H(y))
    m = torch.tensor(wl.m0, device=cuda_device) * (1 + 0.02 * torch.sign(y[0]))
    assert torch.equal(q.forward_nonlinear(m), o.forward_nonlinear(m))
    assert torch.equal(q.gradient(m, r[0].contiguous()), o.gradient(m, r[0].contiguous()))
