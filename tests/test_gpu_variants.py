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
    near = np.clip(wl.src + [2, 3], 0, np.array(shape) - 1)      # traces that are not zero from the start on
    wl.rec = np.concatenate([near, np.stack([rng.integers(0, n, 60) for n in shape], 1)]).astype(np.int32)
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


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def test_autotuned_group_on_the_one_level_kernels(cuda_device):
    """Models that no cluster holds: kernels picked by timing, the group's sweeps captured as one graph."""
    from paper_1101_3615_gb300 import apply_H_group
    wls = [workload((400, 560), 24, 2, 1), workload((430, 500), 24, 3, 2)]
    dms = [torch.tensor(w.trials, device=cuda_device) for w in wls]
    probes = [probe_of(w, use_graph=1) for w in wls]
    first = apply_H_group(probes, dms)
    assert probes[0].stats()["pipeline_forward"] != 1
    again = apply_H_group(probes, dms)
    for w, d, a, b in zip(wls, dms, first, again):
        assert torch.equal(a, b) and bool(a.abs().max() > 0)
        assert rel(a, probe_of(w, pipeline=0, shot_group=1).apply_H(d)) < 1e-6   # the order of the image sums


@pytest.mark.parametrize("ns,nb", [(6, 1), (6, 3), (32, 1)])
def test_adjoint_with_many_items_gives_identical_bits(cuda_device, ns, nb):
    """Six shots of 306 tiles: more than three items for each of four (three) CTAs per SM of 152 SMs, by
    itself and in a group of two models of half the shots; 32 shots: planes beyond the L2."""
    from paper_1101_3615_gb300 import apply_H_group
    wl, half = workload((531, 531), 20, ns, nb), workload((531, 531), 20, ns // 2, nb)
    y = torch.tensor(wl.trials, device=cuda_device)
    for S in (2, 3):
        one, many = probe_of(wl, pipeline=0, shot_group=1), probe_of(wl, pipeline=S, pipe_rows=1, shot_group=1)
        d = one.apply_F(y)
        assert torch.equal(many.apply_Fadj(d), one.apply_Fadj(d))
        assert torch.equal(many.apply_H(y), one.apply_H(y))
        ref = probe_of(half, pipeline=0, shot_group=1).apply_H(y)
        for o in apply_H_group([probe_of(half, pipeline=S, pipe_rows=1, shot_group=1) for _ in range(2)], [y, y]):
            assert torch.equal(o, ref)
