"""Kernel families and variants of the 2D sweeps on grids with all-interior tiles, bit for bit.

Such tiles (64 x 16R cells away from the sponge) take a path of their own in the pipelined kernels, so a
grid needs at least one: 130 columns beside a narrow sponge always hold one.
"""
import numpy as np
import pytest

from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def workload(shape, nt, ns, nb, pad=5):
    rng = np.random.default_rng(4)
    wl = mini_config(2, shape=shape, nt=nt, ns=1, pad=pad, p=1)
    wl.src = np.stack([rng.integers(0, shape[0], ns), rng.integers(0, shape[1], ns)], 1).astype(np.int32)
    wl.wavelet = (wl.wavelet + 0.1 * rng.standard_normal(nt)).astype(np.float32)
    wl.trials = (rng.standard_normal((nb,) + tuple(shape)) * 0.05 * wl.m0.mean()).astype(np.float32)
    return wl


def probe_of(wl, **options):
    from paper_1101_3615_gb300 import Probe
    p = Probe(wl.m0, wl.h, wl.dt, wl.nt, wl.pad, wl.src, wl.rec, wl.wavelet)
    for k, v in options.items():
        p.set_option(k, v)
    return p


@pytest.mark.parametrize("shape,ns,nb", [((60, 200), 2, 2), ((97, 141), 3, 1)])
def test_interior_tiles_give_identical_bits(cuda_device, shape, ns, nb):
    wl = workload(shape, 80, ns, nb)
    y = torch.tensor(wl.trials, device=cuda_device)
    m = torch.tensor(wl.m0, device=cuda_device) * (1 + 0.02 * torch.sign(y[0]))
    one = probe_of(wl, pipeline=0, shot_group=1)
    ref = [one.apply_F(y), one.forward_nonlinear(m), one.apply_H(y)]
    ref += [one.apply_Fadj(ref[0]), one.gradient(m, ref[0][0].contiguous())]
    for name, options in {"resident": {}, "two levels": dict(tblock=2, pipeline=0, shot_group=1),
                          **{f"ring {S} rows {R}": dict(pipeline=S, pipe_rows=R, shot_group=1)
                             for S in (2, 3) for R in (1, 2)}}.items():
        p = probe_of(wl, **options)
        got = [p.apply_F(y), p.forward_nonlinear(m), p.apply_H(y), p.apply_Fadj(ref[0]),
               p.gradient(m, ref[0][0].contiguous())]
        assert all(torch.equal(a, b) for a, b in zip(got, ref)), name
