"""Counters and times of probe_get_stats on the cluster-resident 2D path, on groups and in 3D.

Counts: a group's are the sum of its models' own; the bytes of a 3D adjoint are its model written out
segment by segment.  Times: a group's cover all of its models, and a group leaves the times of an
earlier call on another of its handles alone (factors of two and more apart, so that timer noise does
not matter).
"""
import math

import numpy as np
import pytest

from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def probe_of(wl, **kw):
    from paper_1101_3615_gb300 import Probe
    return Probe(wl.m0, wl.h, wl.dt, wl.nt, wl.pad, wl.src, wl.rec, wl.wavelet, **kw)


def workload(shape, nt, ns, nb, cfg=3):
    wl = mini_config(cfg, shape=shape, nt=nt, ns=ns, pad=6, p=1)
    rng = np.random.default_rng(2)
    wl.trials = (rng.standard_normal((nb,) + tuple(shape)) * 0.05 * wl.m0.mean()).astype(np.float32)
    return wl


COUNTS = ["cell_updates_forward", "cell_updates_recompute", "cell_updates_adjoint",
          "bytes_forward", "bytes_recompute", "bytes_adjoint"]


@pytest.mark.parametrize("resident", [True, False])
def test_group_counts_are_the_sum_of_its_models(cuda_device, resident):
    from paper_1101_3615_gb300 import apply_H_group
    wls = [workload((61, 45), 90, 3, 1), workload((40, 70), 90, 2, 3)]
    probes = [probe_of(w) for w in wls]
    if not resident:
        for p in probes:
            p.set_option("pipeline", 2)
            p.set_option("shot_group", 2)
    dms = [torch.tensor(w.trials, device=cuda_device) for w in wls]
    solo = []
    for p, d in zip(probes, dms):
        p.apply_H(d)
        solo.append(p.stats())
    apply_H_group(probes, dms)
    s = probes[0].stats()
    assert (s["pipeline_forward"] == 1) == resident
    for k in COUNTS:
        assert s[k] == pytest.approx(sum(x[k] for x in solo), rel=1e-12), k


def test_resident_group_times_cover_every_model(cuda_device):
    from paper_1101_3615_gb300 import apply_H_group
    small, large = workload((30, 30), 300, 1, 1), workload((150, 160), 300, 8, 24)
    ps, pl = probe_of(small), probe_of(large)
    ds, dl = (torch.tensor(w.trials, device=cuda_device) for w in (small, large))
    for p in (ps, pl):
        p.set_option("timing", 1)
    one = dl[:1].contiguous()
    solo, single = [], []
    for _ in range(3):
        pl.apply_H(dl)
        solo.append(pl.stats())
        pl.apply_H(one)
        single.append(pl.stats()["ms_adjoint"])
        apply_H_group([ps, pl], [ds, dl])
    pl.apply_H(one)                       # its times are formed when they are read, after the group call
    apply_H_group([ps, pl], [ds, dl])
    late = pl.stats()["ms_adjoint"]
    g = ps.stats()
    for k in ("ms_forward", "ms_adjoint", "ms_total"):
        assert g[k] > 0.7 * min(s[k] for s in solo), k
    assert min(s["ms_adjoint"] for s in solo) > 2.5 * max(single)
    assert late < 1.5 * max(single)


def test_resident_time_block_is_the_launched_segment(cuda_device):
    wl = workload((50, 60), 200, 2, 2)
    y = torch.tensor(wl.trials, device=cuda_device)
    fresh, used = probe_of(wl), probe_of(wl)
    used.apply_H(y)                       # a workspace with checkpoint segments: shorter launches
    ref = fresh.apply_F(y)
    assert torch.equal(used.apply_F(y), ref)
    for p in (fresh, used):
        s = p.stats()
        assert s["pipeline_forward"] == 1
        assert s["launches_forward"] == 2 * math.ceil((wl.nt - 1) / s["time_block"])


@pytest.mark.parametrize("nt,K", [(40, 0), (32, 5), (20, 1)])
@pytest.mark.parametrize("kahan", [True, False])
@pytest.mark.parametrize("pipeline", [None, 2])
def test_adjoint_3d_bytes(cuda_device, nt, K, kahan, pipeline):
    wl = workload((20, 18, 22), nt, 1, 3, cfg=5)
    wl.src = np.array([[2, 5, 6], [3, 12, 15]], np.int32)
    p = probe_of(wl, ckpt_stride=K, kahan=kahan)
    if pipeline:
        p.set_option("pipeline", pipeline)
    p.apply_H(torch.tensor(wl.trials, device=cuda_device))
    s = p.stats()
    assert s["pipeline_adjoint"] == (pipeline or 4)
    stride = s["ckpt_stride"]
    per_cell = 0.0                        # of one (shot, trial); Dtt and s of a shot are shared by its trials
    for k0 in range(0, nt - 1, stride):
        T = min(stride, nt - 1 - k0)
        touches = math.ceil(T / 3) if not pipeline else T      # image updates of the segment
        per_cell += 12.0 * T + (4.0 + 4.0) * T / 3 + 8.0 * touches
        if kahan:
            per_cell += 20.0 - 4.0        # the fold; a segment image is not read by its first update
    cells = float(np.prod([n + 2 * wl.pad for n in (20, 18, 22)]))
    assert s["bytes_adjoint"] == pytest.approx(cells * 2 * 3 * per_cell, rel=1e-12)
