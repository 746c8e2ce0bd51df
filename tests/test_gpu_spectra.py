"""The spectrum path (observable, transform, shell sums) where its kernels
branch: vector and single-node loads, odd and even rows, rows shorter than a
warp, flat boxes, the self-conjugate planes, many shells, and amplitudes far
outside FP32's squared range.

Reference: numpy's FFT of the observable that the FP64 populations give.
Tolerance: an FP32 transform has a relative error of about 2^-24 log2 N in the
root mean square over all modes; a shell's mean of |F|^2 is held to eight
times twice that, of the largest shell mean (thermal spectra are flat), and
the FP64 one to 1e-12.  FP16 storage is read exactly, so it is held as FP32.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2601_03806_gb300 import flbm
    return flbm


def velocities():
    c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for s in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
            v = [0, 0, 0]
            v[a], v[b] = s
            c.append(tuple(v))
    return np.array(c + [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1),
                         (1, -1, -1)])


def weights(obs):
    c = velocities()
    return [np.ones(27), c.sum(1), (c * c).sum(1), c[:, 0] * c[:, 1] + c[:, 0] * c[:, 2] + c[:, 1] * c[:, 2],
            c[:, 0], c[:, 1], c[:, 2]][obs]


def reference(g, obs, nshell):
    m = np.einsum("i,izyx->zyx", weights(obs), g)
    power = np.abs(np.fft.fftn(m)) ** 2 / m.size
    k = [np.fft.fftfreq(n, 1.0 / n) for n in m.shape]
    n2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    s = np.rint(np.sqrt(n2)).astype(int)
    ok = (n2 > 0) & (s < nshell)
    cnt = np.bincount(s[ok], minlength=nshell)
    return np.bincount(s[ok], power[ok], minlength=nshell) / np.maximum(cnt, 1), cnt


@pytest.mark.parametrize("prec", ["fp32", "fp16", "fp64"])
@pytest.mark.parametrize("shape,nshell,steps", [((32, 32, 32), 17, 0), ((64, 6, 5), 40, 1), ((37, 20, 9), 20, 2),
                                                ((1, 7, 1), 5, 1), ((130, 3, 2), 70, 3), ((2, 66, 35), 40, 0),
                                                ((8, 1, 1), 3, 0), ((100, 64, 3), 3072, 0), ((256, 4, 2), 1, 0)])
def test_spectra_match_numpy(F, prec, shape, nshell, steps):
    nx, ny, nz = shape
    box = F.Lattice(nx, ny, nz, 0.8, 1e-5, seed=5, precision=prec)
    box.init_thermal(3)
    box.step(steps)
    w = np.where(velocities().any(1), 0, 8 / 27.0)
    w = np.array([8 / 27.0, 2 / 27.0, 1 / 54.0, 1 / 216.0])[(velocities() ** 2).sum(1)]
    g = box.get_populations() - w[:, None, None, None]
    tol = 1e-12 if prec == "fp64" else 16 * 2.0 ** -24 * max(1.0, np.log2(box.n))
    for obs in range(7):
        S, cnt = box.structure_factor(obs, nshell)
        So, co = reference(g, obs, nshell)
        assert np.array_equal(cnt, co)
        # the subtraction of w rho0 above leaves 1e-16 of noise in g
        assert np.abs(S - So).max() <= tol * So.max() + 1e-25, (obs, np.abs(S - So).max() / max(So.max(), 1e-300))


@pytest.mark.parametrize("scale", [1e-30, 1e-22, 1.0, 1e12, 1e15])
def test_spectra_at_any_amplitude(F, scale):
    """FP32 squares would overflow or vanish; the sums must not."""
    box = F.Lattice(48, 20, 10, 0.8, 0.0, seed=5)
    g = (np.random.default_rng(1).normal(size=(27, 10, 20, 48)) * scale).astype(np.float32)
    box.set_state(g)
    S, cnt = box.structure_factor(F.FLBM_OBS_RHO, 12)
    So, co = reference(g.astype(float), 0, 12)
    assert np.array_equal(cnt, co)
    assert np.abs(S / So - 1)[co > 0].max() <= 16 * 2.0 ** -24 * 14


def test_a_snapshot_leaves_state_and_repeats(F):
    box = F.Lattice(64, 20, 12, 0.8, 1e-5, seed=1)
    box.init_thermal(2)
    box.step(3)
    g = box.get_state()
    a = [box.structure_factor(o, 9)[0] for o in range(4)]
    b = [box.structure_factor(o, 9)[0] for o in range(4)]
    assert np.array_equal(g, box.get_state())
    # the order of the CTAs' FP64 additions is free
    assert all(np.allclose(x, y, rtol=1e-13, atol=0) for x, y in zip(a, b))
