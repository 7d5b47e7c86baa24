"""The Gram and multiplier kernels of the fit at the edges of their ranges, against the FP64 oracle.

Both routes of the first Gram pass (trial sums per point: several spatial modes; all column pairs
per row: one mode, or too many multipliers to stage), both passes at P = 64 and below, numbers of
points that are no multiple of the staged 32 and 128 rows, 2D and 3D, orders other than -1.
Coefficients: 1e-6 relative to their norm, the bar of the other fit tests (condition numbers here
stay below 1e7, so that FP64 round-off alone gives less than 1e-8).  Preconditioned images: 1e-6,
the rounding of the FP32 output being 6e-8.
"""
import numpy as np
import pytest

from oracle.symbol import Basis as OBasis
from oracle.symbol import fit as ofit
from workloads import mini_config

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MODES2 = [(a, b) for a in range(-3, 4) for b in range(-3, 4)]
MODES3 = [(0, 0, 0), (1, 0, 0), (0, -1, 0), (0, 0, 1)]


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def setup(shape, spatial, angular, nradial, order, fft_pad):
    from paper_1101_3615_gb300 import Basis, Probe
    wl = mini_config(5 if len(shape) == 3 else 1, shape=shape, nt=40, ns=1, pad=4, p=1)
    c_mean = float(np.mean(1 / np.sqrt(wl.m0.astype(np.float64))))
    args = (spatial, angular, nradial, 2 * np.pi * 30.0 / c_mean, order, fft_pad)
    p = Probe(wl.m0, wl.h, wl.dt, wl.nt, wl.pad, wl.src, wl.rec, wl.wavelet)
    return wl, p, Basis(wl.ndim, *args), OBasis(wl.shape, wl.h, *args)


@pytest.mark.parametrize("shape,spatial,angular,nradial,p", [
    ((44, 51), MODES2[:32], [0, 2], 1, 3),             # P = 64, most spatial modes
    ((43, 51), [(0, 0)], [0, 2, -2, 4], 2, 2),         # one mode: all pairs per row
    ((43, 51), [(0, 0), (0, 1)], [0, 2, -2, 4, -4, 6, -6, 8], 3, 2),  # 24 multipliers, P = 48
    ((43, 51), [(0, 0), (0, 1)], [0, 2, -2, 4, -4, 6, -6, 8, -8, 10, -10, 12, -12, 14, -14, 16], 2, 4),  # 32: per row
    ((16, 17), MODES2[20:23], [0], 1, 1),              # fewer points than a full staging round
    ((14, 17, 19), MODES3, [0, 4, 5, 1], 2, 2),        # 3D
])
def test_fit_gram_paths_match_oracle(cuda_device, shape, spatial, angular, nradial, p):
    wl, probe, g, o = setup(shape, spatial, angular, nradial, -1.0, 5)
    c_true = np.random.default_rng(3).standard_normal(g.P)
    xs = np.random.default_rng(4).standard_normal((p,) + tuple(shape)).astype(np.float32)
    ys = np.stack([o.apply(c_true, x.astype(np.float64)) for x in xs]).astype(np.float32)
    c_orc, res_orc, cond = ofit(o, ys, xs)
    assert cond < 1e7
    c, res = probe.fit(g, torch.tensor(ys, device=cuda_device), torch.tensor(xs, device=cuda_device))
    assert rel(c, c_orc) < 1e-6, cond
    assert abs(res - res_orc) < 1e-7


@pytest.mark.parametrize("spatial,angular,nradial,sigma", [
    (MODES2[16:32], [0, 2], 2, 0),          # P = 64, cond 9: refined
    (MODES2[:3], [0, 2, -2, 4], 3, 2),      # cond 1e2
    ([(0, 0)], [0, 2], 7, 0),               # cond 4e2, one spatial mode
    ([(0, 0), (1, 0)], [0, 2], 8, 3),       # cond 2e5: the reorthogonalising pass
    ([(0, 0), (1, 0)], [0, 2], 10, 3),      # cond 1e6
    ([(0, 0)], [0, 2], 14, 3),              # cond 2e7
])
def test_fit_refinement_has_the_accuracy_of_qr(cuda_device, spatial, angular, nradial, sigma):
    """Targets that the basis cannot fit (residual of the size of the target) and columns of growing
    condition number: the coefficients against Householder QR within the perturbation bound of the
    least-squares problem, eps cond (2 + cond |r| / (|A| |c|)) with eps = 1e-14 (columns from another FFT)."""
    from scipy.ndimage import gaussian_filter
    shape = (43, 51)
    wl, probe, g, o = setup(shape, spatial, angular, nradial, -1.0, 5)
    xs = np.random.default_rng(4).standard_normal((2,) + shape)
    if sigma:
        xs = np.stack([gaussian_filter(x, sigma) for x in xs])
    xs = xs.astype(np.float32)
    A = np.concatenate([o.columns(x.astype(np.float64)) for x in xs])
    ys = (np.random.default_rng(5).standard_normal((2,) + shape) * np.linalg.norm(A, axis=1).mean()).astype(np.float32)
    c_orc, res_orc, cond = ofit(o, ys, xs)
    c, res = probe.fit(g, torch.tensor(ys, device=cuda_device), torch.tensor(xs, device=cuda_device))
    r = res_orc * np.linalg.norm(ys.astype(np.float64))
    bound = 1e-14 * cond * (2 + cond * r / (np.linalg.norm(A, 2) * np.linalg.norm(c_orc)))
    assert rel(c, c_orc) < bound, (cond, bound)
    assert abs(res - res_orc) < 1e-12


@pytest.mark.parametrize("order", [-1.0, 0.0, 0.5])
@pytest.mark.parametrize("shape,spatial,angular,nradial", [
    ((33, 40), MODES2[:6], [0, 2, -2, 7, -5], 5),
    ((33, 40), [(0, 0)], [3], 1),
    ((33, 40), MODES2[:9], [0, -4], 11),
    ((12, 15, 16), MODES3, [0, 1, 2, 3, 4, 5], 3),
])
def test_precond_spectra_match_oracle(cuda_device, shape, spatial, angular, nradial, order):
    wl, probe, g, o = setup(shape, spatial, angular, nradial, order, 3)
    c = np.random.default_rng(8).standard_normal(g.P)
    img = np.random.default_rng(9).standard_normal(shape).astype(np.float32)
    got = probe.apply_precond(g, c, torch.tensor(img, device=cuda_device)).cpu().numpy()
    assert rel(got, o.apply(c, img.astype(np.float64))) < 1e-6


@pytest.mark.parametrize("q", [2**31 - 1, -2**31 + 1, -2**31])
def test_angular_indices_at_the_ends_of_their_type(cuda_device, q):
    """2D angular indices are not bounded.  The angle of a bin is known to 2**-52 of itself, so its multiple by
    2**31 to about 1e-6; twenty times that for the roundings of 31 squarings and of the oracle's product."""
    wl, probe, g, o = setup((33, 40), [(0, 0)], [q], 2, -1.0, 3)
    c = np.random.default_rng(8).standard_normal(g.P)
    img = np.random.default_rng(9).standard_normal((33, 40)).astype(np.float32)
    got = probe.apply_precond(g, c, torch.tensor(img, device=cuda_device)).cpu().numpy()
    assert rel(got, o.apply(c, img.astype(np.float64))) < 2e-5


@pytest.mark.parametrize("spatial,angular,nradial,sigma", [
    ([(0, 0), (1, 0)], [0, 2], 8, 3),       # cond 2e5
    ([(0, 0)], [0], 14, 2),                 # cond 4e6
    ([(0, 0)], [0, 2], 13, 3),              # cond 7e6
    ([(0, 0), (0, 1)], [0], 14, 3),         # cond 1e7
])
def test_fit_of_targets_in_the_dominant_direction(cuda_device, spatial, angular, nradial, sigma):
    """Targets A v_1 (v_1 the first right singular vector) on ill-conditioned columns: the misfit of the
    first solution is then small however large its error is along the other singular vectors, so it says
    nothing about the condition.  Bound: as in test_fit_refinement_has_the_accuracy_of_qr."""
    from scipy.ndimage import gaussian_filter
    shape = (43, 51)
    wl, probe, g, o = setup(shape, spatial, angular, nradial, -1.0, 5)
    xs = np.random.default_rng(4).standard_normal((2,) + shape)
    xs = np.stack([gaussian_filter(x, sigma) for x in xs]).astype(np.float32)
    A = np.concatenate([o.columns(x.astype(np.float64)) for x in xs])
    ys = (A @ np.linalg.svd(A, full_matrices=False)[2][0]).reshape((2,) + shape).astype(np.float32)
    c_orc, res_orc, cond = ofit(o, ys, xs)
    c, res = probe.fit(g, torch.tensor(ys, device=cuda_device), torch.tensor(xs, device=cuda_device))
    r = res_orc * np.linalg.norm(ys.astype(np.float64))
    bound = 1e-14 * cond * (2 + cond * r / (np.linalg.norm(A, 2) * np.linalg.norm(c_orc)))
    assert rel(c, c_orc) < bound, (cond, bound)


def test_fits_from_two_threads(cuda_device):
    """Handles of their own, streams of their own, staged factors of different size: the same results as alone."""
    import threading
    todo, errors = [], []
    for spatial, angular, nradial in (([(0, 0), (0, 1)], [0, 2, -2, 4, -4, 6, -6, 8], 3), ([(0, 0), (0, 1)], [0], 2)):
        wl, probe, g, o = setup((24, 27), spatial, angular, nradial, -1.0, 2)
        xs = np.random.default_rng(4).standard_normal((2, 24, 27)).astype(np.float32)
        ys = np.random.default_rng(5).standard_normal((2, 24, 27)).astype(np.float32)
        xs, ys = torch.tensor(xs, device=cuda_device), torch.tensor(ys, device=cuda_device)
        todo.append((probe, g, ys, xs, probe.fit(g, ys, xs)[0]))
    torch.cuda.synchronize()

    def work(probe, g, ys, xs, ref):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    assert np.array_equal(probe.fit(g, ys, xs)[0], ref)
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=t) for t in todo]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
