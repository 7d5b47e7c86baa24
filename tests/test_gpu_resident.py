"""The cluster-resident 2D kernels against the one-level kernels, bit for bit.

Both evaluate every cell update in the same order, so the fields, the traces and (with one shot per
image) the images are the same bits.  Grids at the edges of the resident kernels' range: strips of
four rows, one CTA, row blocks that do not fill the strip, widths that are no multiple of four, no
sponge, a source and receivers in strip corners, segments of one level and of the whole recording.
Every case is one that the library's estimate gives to the resident kernels.
"""
import numpy as np
import pytest

from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # interior shape, pad, nt, checkpoint stride, shots, trials
    ((37, 53), 5, 61, 0, 3, 3),
    ((6, 9), 0, 30, 0, 1, 1),          # one CTA, no sponge
    ((16, 7), 0, 26, 5, 2, 2),         # strips of four rows, no sponge
    ((17, 130), 1, 40, 39, 2, 1),      # one segment
    ((129, 66), 9, 37, 5, 2, 1),
    ((203, 317), 17, 41, 20, 3, 1),
    ((201, 241), 20, 40, 0, 6, 1),     # clusters of nine CTAs on the GB300: strips of unequal height
    ((61, 200), 3, 40, 19, 9, 3),      # more fields than clusters at once; a last segment of one level
]


def workload(shape, pad, nt, ns, nb, seed=3):
    rng = np.random.default_rng(seed)
    wl = mini_config(2, shape=shape, nt=nt, ns=ns, pad=pad, p=1)
    nz, nx = shape
    rec = np.stack([rng.integers(0, nz, 50), rng.integers(0, nx, 50)], 1).astype(np.int32)
    wl.rec = np.concatenate([rec, rec[:7], [[0, 0], [nz - 1, nx - 1]]]).astype(np.int32)
    src = np.stack([rng.integers(0, nz, ns), rng.integers(0, nx, ns)], 1).astype(np.int32)
    src[0] = (nz - 1, 0)
    wl.src = src
    wl.wavelet = (wl.wavelet + rng.standard_normal(nt).astype(np.float32) * 0.1).astype(np.float32)
    wl.trials = (rng.standard_normal((nb,) + tuple(shape)) * 0.05 * wl.m0.mean()).astype(np.float32)
    return wl


def probes(wl, K, snap, kahan=True):
    from paper_1101_3615_gb300 import Probe
    out = []
    for resident in (True, False):
        p = Probe(wl.m0, wl.h, wl.dt, wl.nt, wl.pad, wl.src, wl.rec, wl.wavelet, snapshot_dtype=snap, kahan=kahan,
                  ckpt_stride=K)
        if not resident:
            p.set_option("pipeline", 0)
            p.set_option("shot_group", 1)
        out.append(p)
    return out


@pytest.mark.parametrize("shape,pad,nt,K,ns,nb", CASES)
@pytest.mark.parametrize("snap,kahan", [("fp32", True), ("bf16", False), ("fp16", True)])
def test_resident_kernels_give_identical_bits(cuda_device, shape, pad, nt, K, ns, nb, snap, kahan):
    wl = workload(shape, pad, nt, ns, nb)
    res, one = probes(wl, K, snap, kahan)
    y = torch.tensor(wl.trials, device=cuda_device)
    d = one.apply_F(y)
    assert torch.equal(res.apply_F(y), d)
    assert res.stats()["pipeline_forward"] == 1
    r = d + torch.randn(d.shape, device=cuda_device, generator=torch.Generator(cuda_device).manual_seed(1)) * d.std()
    img = one.apply_Fadj(r)
    assert torch.equal(res.apply_Fadj(r), img)
    hy = one.apply_H(y)
    assert torch.equal(res.apply_H(y), hy)
    m = torch.tensor(wl.m0, device=cuda_device) * (1 + 0.02 * torch.sign(y[0]))
    dn = one.forward_nonlinear(m)
    assert torch.equal(res.forward_nonlinear(m), dn)
    g = one.gradient(m, r[0].contiguous())
    assert torch.equal(res.gradient(m, r[0].contiguous()), g)


def test_resident_waves_graph_and_group(cuda_device):
    """Several shot waves, a captured graph, and models of different size in one call."""
    from paper_1101_3615_gb300 import apply_H_group
    wl = workload((45, 70), 6, 50, 5, 2)
    res, one = probes(wl, 0, "fp32")
    y = torch.tensor(wl.trials, device=cuda_device)
    ref = one.apply_H(y)
    assert torch.equal(res.apply_H(y), ref)
    res.set_option("use_graph", 1)
    for _ in range(2):
        assert torch.equal(res.apply_H(y), ref)
    waves = probes(wl, 0, "fp32")[0]
    waves.set_option("shot_wave", 2)
    got = waves.apply_H(y)
    assert float((got - ref).norm() / ref.norm()) < 1e-6   # images of two waves added up
    wl2 = workload((30, 41), 6, 50, 2, 3, seed=8)
    p1, p2 = probes(wl, 0, "fp32")[0], probes(wl2, 0, "fp32")
    y2 = torch.tensor(wl2.trials, device=cuda_device)
    a, b = apply_H_group([p1, p2[0]], [y, y2])
    assert torch.equal(a, ref) and torch.equal(b, p2[1].apply_H(y2))
