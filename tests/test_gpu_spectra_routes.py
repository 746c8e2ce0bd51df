"""The two kernels that bin a spectrum into shells, on both sides of the rule
that picks one (rows of 1 to 4 elements, rows of four chunks of 32 elements in
small and large spectra), and the depth of the scan along a row: a whole warp
in one shell (planes far from the origin), lanes of a shell each; |n|^2 in 32 and
in 64 bits.

Reference and tolerance of test_gpu_spectra.py."""
import numpy as np
import pytest

from test_gpu_spectra import reference, velocities

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("shape,nshell,steps", [((1, 9, 8), 6, 0), ((2, 9, 8), 6, 1), ((3, 9, 8), 6, 0),
                                                ((4, 9, 8), 6, 1), ((1, 1, 500), 260, 0), ((500, 1, 1), 260, 1),
                                                ((300, 3, 2), 130, 0), ((300, 40, 40), 100, 0),
                                                ((300, 40, 40), 95, 1), ((64, 4096, 2), 2100, 0),
                                                ((90000, 1, 1), 64, 0), ((100000, 1, 1), 64, 1)])
def test_shell_sums_on_both_routes(prec, shape, nshell, steps):
    from paper_2601_03806_gb300 import flbm as F
    box = F.Lattice(*shape, 0.8, 1e-5, seed=5, precision=prec)
    box.init_thermal(3)
    box.step(steps)
    w = np.array([8 / 27.0, 2 / 27.0, 1 / 54.0, 1 / 216.0])[(velocities() ** 2).sum(1)]
    g = box.get_populations() - w[:, None, None, None]
    tol = 1e-12 if prec == "fp64" else 16 * 2.0 ** -24 * np.log2(box.n)
    for obs in (0, 3):
        S, cnt = box.structure_factor(obs, nshell)
        So, co = reference(g, obs, nshell)
        assert np.array_equal(cnt, co)
        assert np.abs(S - So).max() <= tol * So.max() + 1e-25
    box.close()
